// The end of a call on the two spread kernels: the outputs of a cluster's CTAs joined, normalised and written, or, with several groups of
// blocks per pair, left in the workspace for the group that arrives last.
//
// What has nothing to say carries (maximum -inf, sum 0, outputs 0): a CTA without text rows, a group or sequence without blocks.  A NaN logit
// leaves a maximum alone (fmaxf drops it) and shows in sum and outputs, so the maximum never decides whether a part counts: each is weighed
// with a finite factor, 0 * 0 for an empty one, 0 * NaN for a NaN one, and a row is zero only where the sum of all parts is.
#pragma once

#include "kvc_fused.cuh"
#include "kvc_spread.cuh"

namespace kvc {

// 2^(x - mx) for a part whose maximum is x where mx is the largest of all: 0 for x = -inf, also where all are
__device__ __forceinline__ float spread_weight(float x, float mx) { return x == -INFINITY ? 0.f : fast_exp2(x - mx); }
__device__ __forceinline__ float spread_ratio(float num, float den) { return den == 0.f ? num : num / den; }

// For CTA `rank` of the cluster of a pair's group rg (C = 2^lc CTAs, dc = 2^ld = 128 / C channels each), with THREADS threads: ystat [C][16]
// (reference maximum, text sum) and yrecv [C][G][dc] of the cluster's CTAs, hstat [16] (maximum, sum) of the vision logits, mus: the CTA's part
// of mu.  flag: a word of shared memory that is free by now; sync(): a barrier of these threads.  C, G, ld and dc come from the kernel, which
// has them in registers (formed anew from the arguments, 32 calls of 1 x 5 blocks of n = 576, 32/32 heads, took 410 us instead of 405).
template <int THREADS, typename Args, typename Sync>
__device__ __forceinline__ void spread_end(const Args& a, int C, int G, int ld, int dc, int tid, int pair, int unit, int rg, int rank,
                                           const float2* ystat, const float* yrecv, const float2* hstat, const float* mus, int* flag, Sync&& sync) {
#pragma unroll 1
  for (int i = tid; i < G * dc; i += THREADS) {
    const int g = i >> ld, d = i & (dc - 1);
    float mx = -INFINITY, num = 0.f, den = 0.f;
#pragma unroll 2
    for (int c = 0; c < C; ++c) mx = fmaxf(mx, ystat[c * 16 + g].x);
#pragma unroll 2
    for (int c = 0; c < C; ++c) {
      const float2 t = ystat[c * 16 + g];
      const float f = spread_weight(t.x, mx);
      num = fmaf(f, yrecv[(c * G + g) * dc + d], num);
      den = fmaf(f, t.y, den);
    }
    const float2 v = hstat[g];
    if (v.y != 0.f) {                                          // (mu is no part of a row without blocks)
      const float f = spread_weight(v.x, mx) * v.y;
      den += f;
      num = fmaf(f, mus[d], num);
    }
    if (a.nrg == 1) {
      store_elem(a.out + ((size_t)pair * G + g) * D + rank * dc + d, spread_ratio(num, den));
    } else {
      a.py[((size_t)unit * G + g) * D + rank * dc + d] = num;
      if (d == 0) a.pml[(((size_t)pair * C + rank) * a.nrg + rg) * G + g] = make_float2(mx, den);
    }
  }
  if (a.nrg > 1) {
    // the last group's CTA `rank` to arrive merges their channels
    __threadfence();
    sync();
    if (tid == 0) *flag = arrive_is_last(&a.cnt[pair * C + rank], a.token, a.nrg) ? 1 : 0;
    sync();
    if (*flag) {
      __threadfence();
#pragma unroll 1
      for (int i = tid; i < G * dc; i += THREADS) {
        const int g = i >> ld, d = i & (dc - 1);
        const float2* ml = a.pml + ((size_t)pair * C + rank) * a.nrg * G + g;
        const float* yp = a.py + ((size_t)pair * a.nrg * G + g) * D + rank * dc + d;
        float mx = -INFINITY, num = 0.f, den = 0.f;
#pragma unroll 4
        for (int p = 0; p < a.nrg; ++p) mx = fmaxf(mx, __ldcg(ml + p * G).x);
#pragma unroll 4
        for (int p = 0; p < a.nrg; ++p) {
          const float2 t = __ldcg(ml + p * G);
          const float f = spread_weight(t.x, mx);
          num = fmaf(f, __ldcg(yp + (size_t)p * G * D), num);
          den = fmaf(f, t.y, den);
        }
        store_elem(a.out + ((size_t)pair * G + g) * D + rank * dc + d, spread_ratio(num, den));
      }
    }
  }
}

}  // namespace kvc
