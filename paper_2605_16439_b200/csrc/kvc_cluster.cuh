// One-kernel bf16 decode path for blocks whose expansions fill tensor-core tiles ("cluster" path): Algorithm 1 for a KV head and
// up to 128 expansion rows (sequence, block, query head) at a time, by a cluster of NS CTAs that share the n axis.
//   step 1   the CTAs of the cluster score the unit's key tiles (64 rows, dealt one by one) and leave S in the workspace
//   step 2   each CTA: L[128 x its columns] = S theta[h] on tcgen05, logits in tensor memory
//   softmax  P = 2^(L - the row's maximum over its columns), the next A operand, in shared memory
//   step 3   each CTA: Wp[128 x m] = P U[h]^T over its columns, partial weights to the workspace with (maximum, sum) per row
//   step 4   the CTAs stream the unit's value tiles (in contiguous runs per warp group), joining the partial weights while the
//            products' B operand is built; a partial (max, sum, y) per (run, sequence)
//   text     (sequence, KV head, chunk of text rows) items, a warp each, on the SMs that have no unit (and after the units)
// The last partial of a (sequence, KV head) to arrive merges them all and writes the output.  S and Wp are a few MB that one
// cluster writes and reads back through L2 between cluster-wide mbarriers; nothing else leaves the SM.
#pragma once

#include "kvc_tma.cuh"
#include "kvc_internal.cuh"

namespace kvc {

constexpr int CL_GROUPS = 3;                       // warp groups of four
constexpr int CL_WARPS = 4 * CL_GROUPS;            // consumer warps
constexpr int CL_CONS = CL_WARPS * 32;
constexpr int CL_THREADS = (CL_WARPS + 2) * 32;    // + MMA issue, + TMA producer
constexpr int CL_ROWS = 128;                       // expansion rows of a unit
constexpr int CL_TILE = 64;                        // key / value rows per tile
constexpr uint32_t CL_HALF = CL_TILE * 128;        // one 64-channel half of a tile
constexpr uint32_t CL_TILE_BYTES = 2 * CL_HALF;
constexpr uint32_t CL_DUE = CL_GROUPS * 16384, CL_W_TAIL = CL_DUE + 512;      // in the region of P while values are summed: behind the groups' reductions
constexpr uint32_t CL_P_BYTES = 65536;             // probabilities; queries, weight staging and the warps' parked accumulators in turn
constexpr int CL_K_SLOTS = 3 * CL_GROUPS, CL_V_SLOTS = 3 * CL_GROUPS, CL_X_SLOTS = 6;      // upper bounds of the rings' slots
constexpr int CL_MAX_NS = 8;
constexpr int CL_MAX_RAGGED_B = 512;
constexpr int CL_TEXT_SLOTS = 4;                   // 16-row pieces in flight per warp of the text part
constexpr int CL_TEXT_CHUNK = 128;                 // text rows per item (more where a pair has as many items as it may)

struct ClusterPlan {
  int ok;
  int units;             // work units of the call
  int terms;             // bf16 terms of S and P
  int NS;                // CTAs per cluster
  int ncl;               // clusters of the grid
  int ucl;               // the first ucl of them take units
  int cap;               // units per KV head that fit in one wave beside the text
  int rbmax;             // blocks per unit that fit 128 rows
  int nu_max;            // most units per KV head any block count up to B R gives
  int ncg;               // 64-column groups of the n axis
  int ms;                // pitch of S and Wp rows, elements
  int nk1;               // 64-row chunks of the m axis
  int npass, prow, nbox, brow;   // passes over the weights (<= 512 columns each), boxes of brow rows of U
  int vt;                // 64-row tiles per block
  int srows;             // expansion rows of a unit: rows of S and W in the workspace, and of S loaded per chunk
  int nK, nX, nV;        // slots of the key ring, the expansion ring and the value ring
  int nwp;                                             // weight slices of the value ring kept in the region of P
  uint32_t x_bytes, s_bytes, w_off, w_bytes, w_tx;     // slot sizes (w_tx: bytes of a slice); the value ring's weights lie behind its tiles
  uint32_t tab_off, pre_off;
  size_t smem;
  int tc, nct;           // text rows per item, items per (sequence, KV head)
  long long text_items, text_ded;                // items, and how many of them the clusters without units take
};

struct ClusterWs {
  size_t off_S, off_W, off_py, off_pml, off_cnt;
  size_t unit_slots;
  size_t bytes;
};

// units of a KV head with nb blocks: as many as fit one wave (never more than blocks), or as few as 128 rows allow
struct UnitSplit { int nu, rb; };
__host__ __device__ __forceinline__ UnitSplit split_units(int nb, int rbmax, int cap) {
  UnitSplit s{0, 1};
  if (nb <= 0) return s;
  int nu = (nb + rbmax - 1) / rbmax;
  if (nu < cap) nu = cap < nb ? cap : nb;
  s.rb = (nb + nu - 1) / nu;
  s.nu = (nb + s.rb - 1) / s.rb;
  return s;
}

int cluster_terms(const kvc_layer* L);                 // bf16 terms of the scores and probabilities (1, 2)
ClusterPlan plan_cluster(const kvc_layer* L, int B, int R, int T, bool ragged);
ClusterWs cluster_ws(const kvc_layer* L, const ClusterPlan& p, int B);
size_t cluster_ws_bytes(const kvc_layer* L, int B, int R, int T_cap);     // for uniform and ragged calls alike; 0 if the path never applies
cudaError_t launch_cluster(const kvc_layer* L, const DecodeArgs& a, const ClusterPlan& p, char* ws, cudaStream_t st, bool* encoded);

struct ClusterArgs {
  const __nv_bfloat16* q;
  const __nv_bfloat16* mu;
  const __nv_bfloat16 *Kc, *Vc, *theta, *U;      // for L2 prefetches
  int theta_np, U_np;    // pitches of their rows
  __nv_bfloat16* out;
  __nv_bfloat16* S;      // [ucl][planes][srows][ms]
  float* W;              // [ucl][NS][srows][ms] partial weights
  float* py;             // [slots][G][D] partials: one per (piece, sequence) of the units, then (from tslot0) [B*H_kv][nct] of the text
  float2* pml;           // [slots][G] (maximum in log2 units, sum)
  int tslot0;
  unsigned long long* cnt;   // [B*H_kv] arrival words
  unsigned int token;
  int* status;
  const int* R_b;
  const int* T_b;
  int early;
  int B, H_kv, G, R, m, n, T;
  int NS, ncl, ucl, cap, rbmax, ncg, ms, nk1, npass, prow, nbox, brow, vt, srows, nK, nX, nV;
  int nwp;
  uint32_t x_bytes, s_bytes, w_off, w_bytes, w_tx, tab_off, pre_off;
  int tc, nct;
  int text_items, text_ded;
};

}  // namespace kvc
