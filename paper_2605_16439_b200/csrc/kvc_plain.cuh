// Plain bf16 decode attention over rows stored verbatim (uncompressed K/V, the text rows alone, the stores of ratio 0), one kernel
// (kvc_plain.cu).  The rows of a (sequence, KV head) are steps of 16 (the vision rows' first, then the text rows'); the steps of all
// pairs form one list that is dealt in equal contiguous runs to the CTAs.
#pragma once

#include "kvc_tma.cuh"
#include "kvc_internal.cuh"

namespace kvc {

constexpr int PN_ROWS = 16;                       // rows per step: a 4 KB piece of K and one of V
constexpr uint32_t PN_PIECE = PN_ROWS * 256u;
constexpr int PN_WARPS = 12;
constexpr int PN_MAX_PARTS = 34;                  // CTAs that can share a (sequence, KV head)

struct PlainPlan {
  int ok;
  int steps_a, spp;        // steps of the leading (vision) rows; of all rows of a pair
  long long total;         // steps of all pairs
  int grid, slots;         // CTAs; pieces in flight per warp
  uint32_t off_red;
  size_t smem;
};

struct PlainWs { size_t off_py, off_pml, off_cnt, bytes; };

PlainPlan plan_plain(const kvc_layer* L, int B, int S0, int T);
PlainWs plain_ws(const kvc_layer* L, int B);
cudaError_t launch_plain(const kvc_layer* L, const DecodeArgs& a, const PlainPlan& p, char* ws, cudaStream_t st, bool* encoded);

struct PlainArgs {
  const __nv_bfloat16* q;
  __nv_bfloat16* out;
  float* py;               // [B*H_kv][slots][G][D]
  float2* pml;             // [B*H_kv][slots][G]  (maximum in log2 units, sum)
  unsigned long long* cnt; // [B*H_kv] arrival words
  unsigned int token;
  int* status;
  int G, S0, T, steps_a, spp, slots;
  long long total;
  uint32_t off_red;
};

}  // namespace kvc
