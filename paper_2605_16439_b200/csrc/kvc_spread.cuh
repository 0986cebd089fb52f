// One-kernel bf16 decode path for small calls ("spread" path): every (sequence, KV head) is served by a cluster of C CTAs that share
// its retained rows and its columns of the n axis, so that a call with few pairs still has most SMs loading.  A sequence's blocks may be split
// into groups with a cluster each, whose outputs meet in the workspace.
//   step 1   CTA c scores its slice of the retained key rows (16-row granules) of every block; the slices of S go to all peers
//   step 2   L[rows x its columns] = S theta[h] on mma.sync, logits in registers; P = 2^(L - the row's maximum over its columns)
//   step 3   Wp = P U[h]^T over its columns; the partial weights of a granule go to the CTA that owns the granule's value rows
//   text     its share of the text rows, 16 at a time per warp, flash-style, while statistics or partial weights travel
//   step 4   y += W Vt over its slice of the value rows, the C partial weights joined on the fly
//   end      the CTAs' outputs meet by ranges of the head dimension: CTA c normalises and writes 128 / C columns
// Everything the CTAs exchange goes through distributed shared memory (bulk copies and st.async, completion on mbarriers); nothing but
// the result, the status word and the groups' partial outputs are written to global memory.
#pragma once

#include "kvc_tma.cuh"
#include "kvc_internal.cuh"

namespace kvc {

constexpr int SPR_WARPS = 16;                         // consumer warps
constexpr int SPR_CONS = SPR_WARPS * 32;
constexpr int SPR_THREADS = SPR_CONS + 32;            // + TMA producer
constexpr int SPR_MAX_C = 8;
constexpr int SPR_MAX_SLOTS = 24;
constexpr int SPR_MAX_NRG = 8;
constexpr int SPR_MAX_WAVES = 4;
constexpr uint32_t SPR_QPITCH = 272;                  // bytes per staged query row (conflict-free ldmatrix)
constexpr int SPR_YLD = 132;                          // pitch of a head's row in the reduction over the warps

struct SpreadPlan {
  int ok;
  int nrg, rg;           // groups of blocks per (sequence, KV head), blocks of a group
  int C;                 // CTAs per group
  int waves;             // of clusters
  int nt;                // 8-row tiles of expansion rows (1, 2, 4, 6, 8)
  int terms;             // bf16 terms of S and P
  int ng, gs;            // 16-row granules of the m axis, and the most of them a CTA has
  int ncg, gw;           // 16-column groups of the n axis, and the most of them a CTA has
  int nsub, gsub, wbox;  // boxes per row of a parameter piece, column groups per box, columns of a box (an odd multiple of 8)
  int pg, npp;           // granules per parameter piece, pieces over the m axis
  int kg, bpp;           // granules and blocks per capsule piece
  int ti;                // 16-row items per text piece
  int slots;
  uint32_t slot_bytes, misc_off, q_off, y_off, s_off, p_off, ring_off;
  size_t smem;
  double us;             // estimate of the call
};

struct SpreadWs {
  size_t off_cnt;        // u64 [B H_kv C] arrival words: CTA c of every group of a pair
  size_t off_py;         // fp32 [B H_kv][nrg][G][D] partial outputs
  size_t off_pml;        // float2 [B H_kv][C][nrg][G] (maximum, sum)
  size_t bytes;
};

SpreadPlan plan_spread(const kvc_layer* L, int B, int R, int T, bool ragged);
SpreadWs spread_ws(const kvc_layer* L, const SpreadPlan& p, int B);
size_t spread_ws_bytes(const kvc_layer* L, int B, int R);     // 0 if the path never applies
bool spread_may_serve(const kvc_layer* L);
cudaError_t launch_spread(const kvc_layer* L, const DecodeArgs& a, const SpreadPlan& p, char* ws, cudaStream_t st, bool* encoded);

// the same for fp32 storage (kvc_spread_f32.cu); of the plan ok, nrg, rg, C, waves and us are set
bool spread_f32_may_serve(const kvc_layer* L);
SpreadPlan plan_spread_f32(const kvc_layer* L, int B, int R, int T);
size_t spread_f32_ws_bytes(const kvc_layer* L, int B, int R);
cudaError_t launch_spread_f32(const kvc_layer* L, const DecodeArgs& a, const SpreadPlan& p, char* ws, cudaStream_t st);

struct SpreadArgs {
  const __nv_bfloat16* q;
  const __nv_bfloat16* mu;
  __nv_bfloat16* out;
  float* py;             // (see SpreadWs)
  float2* pml;
  unsigned long long* cnt;
  unsigned int token;
  int* status;
  const int* R_b;        // per-sequence block counts (<= R) and text lengths (<= T), device arrays; nullptr: R and T for all
  const int* T_b;
  int early;             // 1: capsule rows may be loaded before the stream's previous kernel has finished (see kvc.h)
  int B, H_kv, G, R, m, n, T, nrg, rg;
  int lc, ng, gs, ncg, gw, nsub, gsub, wbox, pg, npp, kg, bpp, ti, slots;      // lc: log2 of the CTAs per cluster
  uint32_t slot_bytes, misc_off, q_off, y_off, s_off, p_off, ring_off;
};

}  // namespace kvc
