// Spread decode kernel (see kvc_spread.cuh) and its host side.
//
// Bound: a chain of dependent steps, four of them exchanges within a cluster of 0.5-1 us; the bytes take a tenth to a half of the time.
// Measured on B200, us per call of a captured graph back to back, the path before / this one: 1 x 5 blocks of n = 576, 32/32 heads, 128 text
// rows (the one-kernel path on 32 SMs) 25.0 / 12.3 (32 layers in turn 12.7; its time line: scores until 2.5 us after the previous kernel's end,
// logits 4.2, probabilities 4.9, text 5.3, weights 6.4, at their owners 7.4, values 9.1, out 10.4); 8 x 5 of n = 729, 28/4 heads (the cluster
// path) 36.6 / 26.9; 1 x 5 of 576, 28/4 heads 24.2 / 13.0; 7 x 2 of 576, m = 404, 37.6 / 14.4; 4 x 5 of 1024, m = 103 (three kernels) 20.6 /
// 11.9; 1 x 1 of 576, 8/2 heads, 16384 text rows 168 / 19.4.
// Why pieces are few and large: a look at a piece by all warps, with its loops, takes some 200 cycles, issuing one some 300 (pieces of 16 KB,
// 21 of them in the first shape: 19.7 us, of 39 KB: 16.9).  Why every loop that need not be is kept rolled: unrolled, the kernel was 100 to
// 130 KB of code, now 50.
#include <algorithm>

#include "kvc_cluster.cuh"
#include "kvc_split.cuh"
#include "kvc_spread_end.cuh"

namespace kvc {

constexpr float SPR_QSCALE = 0.08838834764831845f * 1.4426950408889634f;      // sigma = 1/sqrt(128), logits in log2 units

struct SpreadBars {
  uint64_t full[SPR_MAX_SLOTS], empty[SPR_MAX_SLOTS];
  uint64_t s, stat, w, y;        // score slices, row statistics, partial weights, partial outputs of the peers have landed
};

// one immediate look (half the time of a try_wait), then the bounded wait
__device__ __forceinline__ bool wait_full(uint64_t* bar, uint32_t parity) { return mbar_test_wait(bar, parity) || mbar_wait_bounded(bar, parity); }

// floats as integers of the same order
__device__ __forceinline__ int ordered(float x) { const int i = __float_as_int(x); return i ^ ((i >> 31) & 0x7fffffff); }
__device__ __forceinline__ float unordered(int i) { return __int_as_float(i ^ ((i >> 31) & 0x7fffffff)); }

// The operands of one step of an expansion: A fragments of MG 16-row tiles of the long axis, B fragments of TN row tiles in PL terms
template <int MG, int TN, int PL>
struct SprFrags {
  static constexpr int NP = (TN + 1) / 2;      // ldmatrix pairs of row tiles (the last may be one tile)
  uint32_t a[MG][4], b[PL][NP][4];
  __device__ __forceinline__ void load_rows(uint32_t at, uint32_t plane, uint32_t pitch) {       // at: with the lane's 16-byte part of a row
    const int lane = threadIdx.x & 31, l7 = lane & 7, lrowB = l7 + (lane >> 4) * 8;
#pragma unroll
    for (int pl = 0; pl < PL; ++pl)
#pragma unroll
      for (int t = 0; t < NP; ++t) {
        if (2 * t + 1 < TN) {
          ldsm_x4(b[pl][t], at + pl * plane + (uint32_t)(t * 16 + lrowB) * pitch);
        } else {
          uint32_t v[2];
          ldsm_x2(v, at + pl * plane + (uint32_t)(t * 16 + l7) * pitch);
          b[pl][t][0] = v[0]; b[pl][t][1] = v[1];
        }
      }
  }
  __device__ __forceinline__ void products(float (&acc)[MG][TN][4]) const {
#pragma unroll
    for (int pl = 0; pl < PL; ++pl)
#pragma unroll
      for (int t = 0; t < TN; ++t)
#pragma unroll
        for (int g = 0; g < MG; ++g) mma_bf16_16816(acc[g][t], a[g], b[pl][t / 2][2 * (t & 1)], b[pl][t / 2][2 * (t & 1) + 1]);
  }
};
// steps of an expansion, the next one's loads in flight where registers allow it
template <int MG, int TN, int PL, typename Load>
__device__ __forceinline__ void spr_steps(int steps, float (&acc)[MG][TN][4], Load&& load) {
  if constexpr (MG * 4 + PL * SprFrags<MG, TN, PL>::NP * 4 <= 16) {
    SprFrags<MG, TN, PL> f0, f1;
    load(f0);
#pragma unroll 1
    for (; steps > 2; steps -= 2) {
      load(f1);
      f0.products(acc);
      load(f0);
      f1.products(acc);
    }
    if (steps > 1) load(f1);
    f0.products(acc);
    if (steps > 1) f1.products(acc);
  } else {
#pragma unroll 1
    for (; steps > 0; --steps) {
      SprFrags<MG, TN, PL> f;
      load(f);
      f.products(acc);
    }
  }
}
template <int MG, int TN>
__device__ __forceinline__ void spr_clear(float (&acc)[MG][TN][4]) {
#pragma unroll
  for (int g = 0; g < MG; ++g)
#pragma unroll
    for (int t = 0; t < TN; ++t)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[g][t][e] = 0.f;
}
// v[2 t + e] of the lanes with one t4 joined over gid: lane (gid, t4) receives value gid (halving the values a lane carries at each step
// takes 7 shuffles; a butterfly per value takes 3 each)
template <bool MAX>
__device__ __forceinline__ float spr_join(float (&v)[8]) {
  const int gid = (threadIdx.x & 31) >> 2;
#pragma unroll
  for (int w = 4; w >= 1; w >>= 1) {
    const bool up = (gid & w) != 0;
#pragma unroll
    for (int i = 0; i < w; ++i) {
      const float out = up ? v[i] : v[i + w], in = up ? v[i + w] : v[i];
      const float got = __shfl_xor_sync(0xffffffffu, out, 4 * w);
      v[i] = MAX ? fmaxf(in, got) : in + got;
    }
  }
  return v[0];
}

// NT: 8-row tiles of expansion rows (row r G + g); NH: 8-head tiles; PL: bf16 terms of S and P
template <int NT, int NH, int PL>
__global__ void __launch_bounds__(SPR_THREADS, 1)
spread_decode_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
                     const __grid_constant__ CUtensorMap tmKt, const __grid_constant__ CUtensorMap tmVt,
                     const __grid_constant__ CUtensorMap tmTh, const __grid_constant__ CUtensorMap tmU,
                     const __grid_constant__ SpreadArgs a) {
  constexpr int RP = NT * 8;                   // expansion rows, padded
  // A warp's tile of the two expansions: MG 16-row tiles of the long axis (columns of theta, rows of U) by TN row tiles.  With more than two
  // row tiles a warp takes half of them for two tiles of the long axis, so that the fragments a step loads serve MG TN products.
  constexpr int MG = NT > 2 ? 2 : 1, NSP = NT > 2 ? 2 : 1, TN = NT / NSP;
  constexpr bool EARLY_TEXT = NT <= 2 && NH == 1;      // the text rows between the two expansions, while the statistics travel: registers allow it
  constexpr int RW = RP + 4;                   // pitch of a partial weight row: its reads hit 32 banks
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* sm = smem_raw + ((1024u - (smem_addr(smem_raw) & 1023u)) & 1023u);
  __shared__ __align__(8) SpreadBars bars;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int C = 1 << a.lc, G = a.G, rank = (int)blockIdx.x & (C - 1), unit = (int)blockIdx.x >> a.lc;
  const int pair = a.nrg > 1 ? unit / a.nrg : unit, rg = unit - pair * a.nrg;    // group of blocks [rg a.rg, ...) of (b, h)
  const int b = pair / a.H_kv, h = pair - b * a.H_kv;
  const bool ragged = a.R_b != nullptr || a.T_b != nullptr;

  // this CTA's granules of the m axis and column groups of the n axis
  const int g0 = rank * a.ng >> a.lc, gown = ((rank + 1) * a.ng >> a.lc) - g0;
  const int cg0 = rank * a.ncg >> a.lc, cown = ((rank + 1) * a.ncg >> a.lc) - cg0;

  int* rowmax = reinterpret_cast<int*>(sm + a.misc_off);                        // [RP]
  float* psum = reinterpret_cast<float*>(rowmax + RP);                          // [SPR_WARPS / NSP][RP]
  float2* stat = reinterpret_cast<float2*>(psum + SPR_WARPS / NSP * RP);        // [C][RP] (maximum, sum), written by the peers
  float2* tstat = stat + SPR_MAX_C * RP;                                        // [SPR_WARPS][16] text (maximum, sum) per warp and head
  float2* hstat = tstat + SPR_WARPS * 16;                                       // [16] vision (maximum, sum) per head
  float2* ystat = hstat + 16;                                                   // [C][16] (reference maximum, text sum), written by the peers
  float* mus = reinterpret_cast<float*>(ystat + SPR_MAX_C * 16);                // [128 / C] this CTA's part of mu
  float* yrecv = reinterpret_cast<float*>(sm + a.y_off);                        // [C][G][128 / C], written by the peers
  const uint32_t spitch = (uint32_t)(a.gs * 16 + 8) * 2u, splane = RP * spitch, sslice = PL * splane;      // S: [C][PL][RP][gs 16 + 8]
  const uint32_t ppitch = (uint32_t)(a.gw * 16 + 8) * 2u, pplane = RP * ppitch;                            // P: [PL][RP][gw 16 + 8]
  const uint32_t s_u = smem_addr(sm + a.s_off), p_u = smem_addr(sm + a.p_off);
  const float* Wr = reinterpret_cast<const float*>(sm + a.s_off);               // [C][gs 16][RW] once S is no longer needed
  unsigned char* ring = sm + a.ring_off;

  const uint32_t kbytes = (uint32_t)(a.kg * 16 * a.bpp) * 256u, pbytes = (uint32_t)(a.nsub * a.pg * 16 * a.wbox) * 2u;
  const int kp = gown > a.kg ? (gown + a.kg - 1) / a.kg : 1;  // capsule pieces per run of blocks
  const int blk = pair * a.R + rg * a.rg;                     // first block in the capsule store
  // blocks of the group in a sequence that has r of them
  auto group_blocks = [&](int r) { return min(max(r - rg * a.rg, 0), a.rg); };
  // this CTA's share of the text rows, in items of 16
  auto text_items = [&](int t, int& i0, int& i1) {
    const uint32_t items = (uint32_t)(t + 15) >> 4, c = (uint32_t)(rg * C + rank), n = (uint32_t)a.nrg << a.lc;
    const uint32_t q = a.nrg == 1 ? items >> a.lc : items / n, rem = items - q * n;
    i0 = (int)(c * q + min(c, rem)); i1 = i0 + (int)(q + (c < rem ? 1u : 0u));
  };
  auto load_capsule = [&](const CUtensorMap* tm, uint32_t slot, int r, int x) {
    tma_load_4d(ring + slot * a.slot_bytes, tm, 0, (g0 + x * a.kg) * 16, 0, blk + r, &bars.full[slot]);
  };
  // Barriers: one thread each (one after the other they would take most of a microsecond).  The producer's lanes set up the ring's slots and
  // fill those that key rows take before anything else happens in the CTA, once the rows are settled (a thread issues a piece only every 300
  // cycles or so).  Not theta's: with the whole ring on its way the stream's previous kernel ends later (32 pairs, 5 blocks of n = 576: 14.0
  // us per call, 13.2 with the key rows alone, 13.3 with nothing this early; 4 pairs of n = 1024: 23.9, 23.9, 24.3).
  int filled = 0;
  if (warp == SPR_WARPS) {
    const int nk = ((group_blocks(a.R) + a.bpp - 1) / a.bpp) * kp;
    if (a.early && !ragged) filled = min(a.slots, nk);
    if (lane < a.slots) {
      mbar_init(&bars.full[lane], 1); mbar_init(&bars.empty[lane], SPR_WARPS);
      fence_mbar_init();
      if (lane < filled) {
        mbar_expect_tx(&bars.full[lane], kbytes);
        const int q = lane / kp;
        load_capsule(&tmK, (uint32_t)lane, q * a.bpp, lane - q * kp);
      }
    }
    __syncwarp();
  } else if (tid < 4) {
    uint64_t* bar = &bars.s + tid;
    mbar_init(bar, 1);
    fence_mbar_init();
    mbar_expect_tx(bar, tid == 0 ? (uint32_t)(C - 1) * sslice : (tid == 1 ? (uint32_t)(C * RP * 8) :
                        (tid == 2 ? (uint32_t)(C * gown * 16 * RP * 4) : (uint32_t)(G * D * 4 + C * G * 8))));
  } else if (tid >= 32 && tid < 32 + RP) {
    rowmax[tid - 32] = (int)0x80000000;
  }
  __syncthreads();
  cluster_arrive();

  if (warp == SPR_WARPS) {
    // =========================================== producer ===========================================
    if (lane == 0) {
      bool ok = true, waited = false;
      uint32_t slot = filled == a.slots ? 0u : (uint32_t)filled, round = filled == a.slots ? 1u : 0u;
      int skip = filled;                                      // pieces that are on their way already
      auto begin = [&](uint32_t bytes) {
        if (round > 0 && !wait_full(&bars.empty[slot], (round & 1u) ^ 1u)) { ok = false; return false; }
        mbar_expect_tx(&bars.full[slot], bytes);
        return true;
      };
      auto end = [&]() { if (++slot == (uint32_t)a.slots) { slot = 0; ++round; } };
      // lengths are inputs like the queries; the capsule rows may be read early once they are settled, the parameters always
      if (ragged || !a.early) { grid_dep_wait(); waited = true; }
      int Re = a.R, Te = a.T;
      if (a.R_b) { const int r = a.R_b[b]; Re = r < 0 ? 0 : (r > a.R ? a.R : r); }
      if (a.T_b) { const int t = a.T_b[b]; Te = t < 0 ? 0 : (t > a.T ? a.T : t); }
      Re = group_blocks(Re);
      auto capsule = [&](const CUtensorMap* tm) {
#pragma unroll 1
        for (int r = 0; r < Re && ok; r += a.bpp)
#pragma unroll 1
          for (int x = 0; x < kp; ++x) {
            if (skip > 0) { --skip; continue; }
            if (!begin(kbytes)) return;
            load_capsule(tm, slot, r, x);
            end();
          }
      };
      auto params = [&](const CUtensorMap* tm) {
#pragma unroll 1
        for (int p = 0; p < a.npp && ok; ++p) {
          if (!begin(pbytes)) return;
#pragma unroll 1
          for (int s = 0; s < a.nsub; ++s)
            tma_load_3d(ring + slot * a.slot_bytes + (uint32_t)(s * a.pg * 16 * a.wbox) * 2u, tm, (cg0 + s * a.gsub) * 16, p * a.pg * 16, h,
                        &bars.full[slot]);
          end();
        }
      };
      auto text = [&]() {
        int i0, i1;
        text_items(Te, i0, i1);
#pragma unroll 1
        for (int i = i0; i < i1 && ok; i += a.ti) {
          if (!begin((uint32_t)a.ti * 8192u)) return;
          tma_load_5d(ring + slot * a.slot_bytes, &tmKt, 0, i * 16, 0, h, b, &bars.full[slot]);
          tma_load_5d(ring + slot * a.slot_bytes + (uint32_t)a.ti * 4096u, &tmVt, 0, i * 16, 0, h, b, &bars.full[slot]);
          end();
        }
      };
      if (Re > 0) {
        capsule(&tmK);
        params(&tmTh);
        if (!EARLY_TEXT) params(&tmU);
      }
      if (!waited) grid_dep_wait();
      text();
      if (Re > 0) {
        if (EARLY_TEXT) params(&tmU);
        capsule(&tmV);
      }
      if (!ok) atomicExch(a.status, (int)KVC_ERR_TIMEOUT);
    }
    __syncwarp();
    cluster_wait();
    cluster_arrive();
  } else {
    // =========================================== consumers ===========================================
    const int gid = lane >> 2, t4 = lane & 3, l7 = lane & 7, lmid = (lane >> 3) & 1, lhi = lane >> 4, lrowB = l7 + lhi * 8, lrowA = l7 + lmid * 8;
    bool dead = false;
    uint32_t slot = 0, par = 0;
    auto acquire = [&]() -> unsigned char* {
      if (!dead && !wait_full(&bars.full[slot], par)) dead = true;
      __syncwarp();
      return ring + slot * a.slot_bytes;
    };
    auto release = [&]() {
      __syncwarp();
      if (lane == 0) mbar_arrive(&bars.empty[slot]);
      if (++slot == (uint32_t)a.slots) { slot = 0; par ^= 1u; }
    };
    auto peer_wait = [&](uint64_t* bar) { if (!dead && !mbar_wait_cluster_bounded(bar, 0u)) dead = true; };

    if (tid < D >> a.lc) mus[tid] = __bfloat162float(a.mu[h * D + rank * (D >> a.lc) + tid]);      // (a parameter)
    // reciprocals for the divisions of small numbers below, made while the previous kernel runs
    const uint32_t inv_full = (65536u + (uint32_t)a.kg - 1u) / (uint32_t)a.kg, cnt_last = (uint32_t)(gown - (kp - 1) * a.kg), inv_last = (65536u + cnt_last - 1u) / cnt_last;
    const float inv_ng = 1.f / (float)a.ng;
    if (tid < 2 * G) prefetch_l2(a.q + ((size_t)pair * G) * D + tid * 64);      // consumes nothing: may run before the wait
    grid_dep_wait();
    grid_dep_launch();
    if (blockIdx.x == 0 && warp == 0) {
      if (lane == 0) *a.status = 0;
      __syncwarp();
      if (ragged)
#pragma unroll 1
        for (int x = lane; x < a.B; x += 32)
          if ((a.R_b && (a.R_b[x] < 0 || a.R_b[x] > a.R)) || (a.T_b && (a.T_b[x] < 0 || a.T_b[x] > a.T))) atomicExch(a.status, (int)KVC_ERR_BOUNDS);
    }
    int Re = a.R, Te = a.T;
    if (a.R_b) { const int r = a.R_b[b]; Re = r < 0 ? 0 : (r > a.R ? a.R : r); }
    if (a.T_b) { const int t = a.T_b[b]; Te = t < 0 ? 0 : (t > a.T ? a.T : t); }
    Re = group_blocks(Re);

    // the pair's queries, an A operand whose rows are the heads: read from shared memory where they are used (held in registers they spill)
#pragma unroll 1
    for (int i = tid; i < 16 * 16; i += SPR_CONS) {
      const int g = i >> 4, c = i & 15;
      *reinterpret_cast<uint4*>(sm + a.q_off + (uint32_t)g * SPR_QPITCH + c * 16u) =
          g < G ? *reinterpret_cast<const uint4*>(a.q + ((size_t)pair * G + g) * D + c * 8) : make_uint4(0, 0, 0, 0);
    }
    const uint32_t q_u = smem_addr(sm + a.q_off) + (uint32_t)lrowA * SPR_QPITCH + (uint32_t)lhi * 16u;
    // 16 key rows (halves of 64 channels `half` bytes apart): c[8-key tile] = logits of (head gid (+8), keys 2 t4, + 1), in log2 units
    auto score16 = [&](uint32_t base, uint32_t half, float (&c)[2][4]) {
      float c2[2][2][4];
#pragma unroll
      for (int x = 0; x < 2; ++x)
#pragma unroll
        for (int nt = 0; nt < 2; ++nt)
#pragma unroll
          for (int e = 0; e < 4; ++e) c2[x][nt][e] = 0.f;
#pragma unroll
      for (int k0 = 0; k0 < 8; k0 += 4) {
        uint32_t qa[4][4], bk[4][4];
#pragma unroll
        for (int x = 0; x < 4; ++x) {
          ldsm_x4(qa[x], q_u + (k0 + x) * 32u);
          ldsm_x4(bk[x], base + (uint32_t)lrowB * 128u + (k0 >> 2) * half + (uint32_t)(((x * 2 + lmid) ^ l7) << 4));
        }
#pragma unroll
        for (int x = 0; x < 4; ++x) {
          mma_bf16_16816(c2[x & 1][0], qa[x], bk[x][0], bk[x][1]);
          mma_bf16_16816(c2[x & 1][1], qa[x], bk[x][2], bk[x][3]);
        }
      }
#pragma unroll
      for (int nt = 0; nt < 2; ++nt)
#pragma unroll
        for (int e = 0; e < 4; ++e) c[nt][e] = (c2[0][nt][e] + c2[1][nt][e]) * SPR_QSCALE;
    };
    float y[8][NH][4];                                        // [16 channels][8 heads]: channels gid, gid + 8, heads 2 t4, + 1
#pragma unroll
    for (int mt = 0; mt < 8; ++mt)
#pragma unroll
      for (int nh = 0; nh < NH; ++nh)
#pragma unroll
        for (int e = 0; e < 4; ++e) y[mt][nh][e] = 0.f;
    float m_run[NH], l_run[NH];                               // of head gid (+ 8)
#pragma unroll
    for (int nh = 0; nh < NH; ++nh) { m_run[nh] = -INFINITY; l_run[nh] = 0.f; }
    auto scale_heads = [&](const float (&f)[NH]) {            // f: of head gid (+ 8)
#pragma unroll
      for (int nh = 0; nh < NH; ++nh) {
        const float f0 = __shfl_sync(0xffffffffu, f[nh], 8 * t4), f1 = __shfl_sync(0xffffffffu, f[nh], 8 * t4 + 4);
#pragma unroll
        for (int mt = 0; mt < 8; ++mt) { y[mt][nh][0] *= f0; y[mt][nh][1] *= f1; y[mt][nh][2] *= f0; y[mt][nh][3] *= f1; }
      }
    };
    // y += (16 value rows)^T w; w[nh]: weights of head gid (+ 8) at rows 2 t4, + 1, 2 t4 + 8, + 9, as two bf16 terms
    auto values16 = [&](uint32_t base, uint32_t half, const float (&w)[NH][4]) {
      uint32_t hi[NH][2], lo[NH][2];
#pragma unroll
      for (int nh = 0; nh < NH; ++nh)
#pragma unroll
        for (int x = 0; x < 2; ++x) {
          hi[nh][x] = pack2_bf16(w[nh][2 * x], w[nh][2 * x + 1]);
          lo[nh][x] = split_lo(w[nh][2 * x], w[nh][2 * x + 1], hi[nh][x]);
        }
#pragma unroll
      for (int m0 = 0; m0 < 8; m0 += 4) {
        uint32_t v[4][4];
#pragma unroll
        for (int x = 0; x < 4; ++x) ldsm_x4_t(v[x], base + (uint32_t)lrowB * 128u + (m0 >> 2) * half + (uint32_t)(((x * 2 + lmid) ^ l7) << 4));
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
          for (int nh = 0; nh < NH; ++nh) mma_bf16_16816(y[m0 + x][nh], v[x], hi[nh][0], hi[nh][1]);
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
          for (int nh = 0; nh < NH; ++nh) mma_bf16_16816(y[m0 + x][nh], v[x], lo[nh][0], lo[nh][1]);
      }
    };
    // this CTA's share of the text rows: 16 at a time, a warp each, flash-style
    auto text_part = [&]() {
      int i0, i1;
      text_items(Te, i0, i1);
      int first = SPR_WARPS - 1 - warp;                       // item of the piece; every sixteenth is this warp's (the last warps have the fewest granules)
#pragma unroll 1
      for (int i = i0; i < i1; i += a.ti) {
        unsigned char* pc = acquire();
        const int cnt = min(a.ti, i1 - i);
        const uint32_t half = (uint32_t)a.ti * 2048u;
#pragma unroll 1
        for (; first < cnt; first += SPR_WARPS) {
          const uint32_t base = smem_addr(pc) + (uint32_t)first * 2048u;
          const int nv = min(16, Te - (i + first) * 16);
          float c[2][4], f[NH], w[NH][4];
          score16(base, half, c);
#pragma unroll
          for (int hr = 0; hr < NH; ++hr) {
            float mx = -INFINITY;
#pragma unroll
            for (int nt = 0; nt < 2; ++nt)
#pragma unroll
              for (int x = 0; x < 2; ++x) {
                float& z = c[nt][2 * hr + x];
                z = nt * 8 + 2 * t4 + x < nv ? z : -INFINITY;
                mx = fmaxf(mx, z);
              }
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
            const float m_new = fmaxf(m_run[hr], mx);         // finite: the item holds at least one row
            f[hr] = fast_exp2(m_run[hr] - m_new);
            m_run[hr] = m_new;
            float ps = 0.f;
#pragma unroll
            for (int nt = 0; nt < 2; ++nt)
#pragma unroll
              for (int x = 0; x < 2; ++x) { const float z = fast_exp2(c[nt][2 * hr + x] - m_new); w[hr][2 * nt + x] = z; ps += z; }
            l_run[hr] = l_run[hr] * f[hr] + ps;
          }
          scale_heads(f);
          const bool ragged_rows = a.T_b != nullptr && nv < 16;
          if (ragged_rows) {
            // rows past the sequence's length may hold anything (rows past T are zero-filled by the copy)
#pragma unroll 1
            for (int x = lane; x < (16 - nv) * 16; x += 32) {
              const int rr = nv + (x >> 4), cc = x & 15;
              *reinterpret_cast<uint4*>(pc + 2u * half + (uint32_t)first * 2048u + (uint32_t)(cc >> 3) * half + (uint32_t)rr * 128u + (uint32_t)(cc & 7) * 16u) =
                  make_uint4(0, 0, 0, 0);
            }
            __syncwarp();
          }
          values16(base + 2u * half, half, w);
          if (ragged_rows) fence_proxy_async();               // the zeroed rows before the next copy into this slot
        }
        first -= cnt;
        release();
      }
#pragma unroll
      for (int nh = 0; nh < NH; ++nh) {
        l_run[nh] += __shfl_xor_sync(0xffffffffu, l_run[nh], 1);
        l_run[nh] += __shfl_xor_sync(0xffffffffu, l_run[nh], 2);
        if (t4 == 0) tstat[warp * 16 + gid + 8 * nh] = make_float2(m_run[nh], l_run[nh]);
      }
    };
    named_barrier_sync(1, SPR_CONS);
    cluster_wait();                                           // the peers' barriers exist

    const int cgl = MG == 2 ? warp & ~1 : warp, hf = NSP == 2 ? warp & 1 : 0;      // step 2: first column group and part of the row tiles
    const bool mine = cgl < cown;
    const int jrow = (hf * TN + (gid >> 1)) * 8 + 2 * t4 + (gid & 1);              // the row whose joined value the lane holds
    const uint32_t wp = (uint32_t)a.wbox * 2u, sub = (uint32_t)(a.pg * 16) * wp;   // pitch and size of a parameter box
    if (Re > 0) {
      // ---------------- step 1: scores of this CTA's key rows ----------------
      {
        int first = warp;                                     // task: (block, granule); every sixteenth is this warp's
#pragma unroll 1
        for (int r0 = 0; r0 < Re; r0 += a.bpp)
#pragma unroll 1
          for (int x = 0; x < kp; ++x) {
            const uint32_t pc = smem_addr(acquire());
            const int cnt = min(a.kg, gown - x * a.kg), tasks = min(a.bpp, Re - r0) * cnt;
            const uint32_t inv = x + 1 < kp ? inv_full : inv_last;      // first / cnt for the few tasks of a piece
#pragma unroll 1
            for (; first < tasks; first += SPR_WARPS) {
              const int bl = (int)((uint32_t)first * inv >> 16), gi = first - bl * cnt, r = r0 + bl;
              const uint32_t half = (uint32_t)a.kg * 2048u;
              float c[2][4];
              score16(pc + (uint32_t)bl * 2u * half + (uint32_t)gi * 2048u, half, c);
              const uint32_t dst = a.s_off + (uint32_t)rank * sslice + (uint32_t)((x * a.kg + gi) * 16 + 2 * t4) * 2u;
#pragma unroll
              for (int hr = 0; hr < NH; ++hr)
                if (gid + 8 * hr < G)
#pragma unroll
                  for (int nt = 0; nt < 2; ++nt) {
                    const uint32_t hi = pack2_bf16(c[nt][2 * hr], c[nt][2 * hr + 1]);
                    unsigned char* d0 = sm + dst + (uint32_t)(r * G + gid + 8 * hr) * spitch + nt * 16u;
                    *reinterpret_cast<uint32_t*>(d0) = hi;
                    if (PL == 2) *reinterpret_cast<uint32_t*>(d0 + splane) = split_lo(c[nt][2 * hr], c[nt][2 * hr + 1], hi);
                  }
            }
            first -= tasks;
            release();
          }
        fence_proxy_async();                                  // the slice before the copies that read it
        named_barrier_sync(1, SPR_CONS);
        if (warp == 0 && lane < C && lane != rank) {
          const uint32_t src = s_u + (uint32_t)rank * sslice;
          bulk_s2peer(map_to_cta(src, (uint32_t)lane), src, sslice, map_to_cta(smem_addr(&bars.s), (uint32_t)lane));
        }
      }
      // ---------------- step 2: logits of this CTA's columns ----------------
      {
        float acc[MG][TN][4];
        spr_clear(acc);
        uint32_t col[MG];
#pragma unroll
        for (int g = 0; g < MG; ++g) {
          const int cg = min(cgl + g, cown - 1), sb = cg >= a.gsub ? 1 : 0;
          col[g] = (uint32_t)sb * sub + (uint32_t)((cg - sb * a.gsub) * 16 + lmid * 8) * 2u + (uint32_t)lrowB * wp;
        }
        int k = 0, src = 0, s_end = a.ng >> a.lc;             // granule k lies in slice src, which ends at s_end
        const uint32_t s0 = s_u + (uint32_t)lmid * 16u + (uint32_t)(hf * TN * 8) * spitch;
        uint32_t sk = s0;
        peer_wait(&bars.s);
        __syncwarp();
#pragma unroll 1
        for (int p = 0; p < a.npp; ++p) {
          uint32_t tp = smem_addr(acquire());
          if (mine) {
            const int k_end = min(a.ng, (p + 1) * a.pg);
            spr_steps<MG, TN, PL>(k_end - k, acc, [&](SprFrags<MG, TN, PL>& x) {
#pragma unroll
              for (int g = 0; g < MG; ++g) ldsm_x4_t(x.a[g], tp + col[g]);
              x.load_rows(sk, splane, spitch);
              tp += 16u * wp;
              const bool next = ++k == s_end;
              src += next ? 1 : 0;
              s_end = next ? (src + 1) * a.ng >> a.lc : s_end;
              sk = next ? s0 + (uint32_t)src * sslice : sk + 32u;
            });
          }
          release();
        }
        // probabilities relative to the row's maximum over this CTA's columns; acc[g][t]: columns gid, gid + 8, rows 8 t + 2 t4, + 1
        bool ok[MG][2];
#pragma unroll
        for (int g = 0; g < MG; ++g)
#pragma unroll
          for (int x = 0; x < 2; ++x) ok[g][x] = cgl + g < cown && (cg0 + cgl + g) * 16 + 8 * x + gid < a.n;
        float v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          v[i] = -INFINITY;
          if (i < 2 * TN)
#pragma unroll
            for (int g = 0; g < MG; ++g)
#pragma unroll
              for (int x = 0; x < 2; ++x) v[i] = fmaxf(v[i], ok[g][x] ? acc[g][(i / 2) % TN][2 * x + (i & 1)] : -INFINITY);
        }
        {
          const float mx = spr_join<true>(v);
          if (mine && (gid >> 1) < TN) atomicMax(&rowmax[jrow], ordered(mx));
        }
        named_barrier_sync(1, SPR_CONS);
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = 0.f;
#pragma unroll
        for (int t = 0; t < TN; ++t) {
          const int2 mi = *reinterpret_cast<const int2*>(&rowmax[(hf * TN + t) * 8 + 2 * t4]);
          const float mx[2] = {unordered(mi.x), unordered(mi.y)};
#pragma unroll
          for (int g = 0; g < MG; ++g)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              acc[g][t][e] = ok[g][e >> 1] ? fast_exp2(acc[g][t][e] - mx[e & 1]) : 0.f;
              v[2 * t + (e & 1)] += acc[g][t][e];
            }
        }
        if (mine) {
          // transposed on the way to shared memory: P's rows are the expansion rows
#pragma unroll
          for (int g = 0; g < MG; ++g) {
            if (g == 1 && cgl + 1 >= cown) break;
            const uint32_t d0 = p_u + (uint32_t)(hf * TN * 8 + l7) * ppitch + (uint32_t)((cgl + g) * 16 + lmid * 8) * 2u;
#pragma unroll
            for (int t = 0; t < TN; t += 2) {
              uint32_t hi[4];
#pragma unroll
              for (int x = 0; x < 4; ++x) {
                const int tt = (t + (x >> 1)) % TN;
                hi[x] = t + (x >> 1) < TN ? pack2_bf16(acc[g][tt][2 * (x & 1)], acc[g][tt][2 * (x & 1) + 1]) : 0u;
              }
              const uint32_t at = d0 + (uint32_t)((t + (t + 1 < TN ? lhi : 0)) * 8) * ppitch;
              if (t + 1 < TN) stsm_x4_t(at, hi); else stsm_x2_t(at, hi[0], hi[1]);
              if (PL == 2) {
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                  const int tt = (t + (x >> 1)) % TN;
                  hi[x] = t + (x >> 1) < TN ? split_lo(acc[g][tt][2 * (x & 1)], acc[g][tt][2 * (x & 1) + 1], hi[x]) : 0u;
                }
                if (t + 1 < TN) stsm_x4_t(at + pplane, hi); else stsm_x2_t(at + pplane, hi[0], hi[1]);
              }
            }
          }
        }
        {
          const float s = spr_join<false>(v);
          if ((gid >> 1) < TN) psum[(NSP == 2 ? warp >> 1 : warp) * RP + jrow] = mine ? s : 0.f;
        }
      }
      named_barrier_sync(1, SPR_CONS);
      if (tid < RP) {
        float s = 0.f;
#pragma unroll
        for (int w = 0; w < SPR_WARPS / NSP; ++w) s += psum[w * RP + tid];
        const float mx = unordered(rowmax[tid]);
        const uint32_t dst = smem_addr(&stat[rank * RP + tid]), bar = smem_addr(&bars.stat);
#pragma unroll 1
        for (int c = 0; c < C; ++c) st_async_f32x2(map_to_cta(dst, (uint32_t)c), mx, s, map_to_cta(bar, (uint32_t)c));
      }
    }
    if (EARLY_TEXT) text_part();
    if (Re > 0) {
      // ---------------- step 3: partial weights over this CTA's columns, sent to the granules' owners ----------------
      bool settled = false;                                   // the statistics of all CTAs: they have read their S, whose memory the weights take
      int first = warp;                                       // task: (MG granules, part of the row tiles)
#pragma unroll 1
      for (int p = 0; p < a.npp; ++p) {
        const uint32_t pc = smem_addr(acquire());
        const int cnt = min(a.pg, a.ng - p * a.pg), tasks = MG == 2 ? (cnt + 1) & ~1 : cnt;
#pragma unroll 1
        for (; first < tasks; first += SPR_WARPS) {
          const int kp0 = MG == 2 ? first & ~1 : first, part = NSP == 2 ? first & 1 : 0;
          float acc[MG][TN][4];
          spr_clear(acc);
          uint32_t up = pc + (uint32_t)(kp0 * 16 + lrowA) * wp + (uint32_t)lhi * 16u;
          const uint32_t up1 = MG == 2 && kp0 + 1 < cnt ? 16u * wp : 0u;                       // the second granule (or the first again)
          uint32_t pk = p_u + (uint32_t)lmid * 16u + (uint32_t)(part * TN * 8) * ppitch;
          int left = a.gsub;
          spr_steps<MG, TN, PL>(cown, acc, [&](SprFrags<MG, TN, PL>& x) {
#pragma unroll
            for (int g = 0; g < MG; ++g) ldsm_x4(x.a[g], up + (g ? up1 : 0u));
            x.load_rows(pk, pplane, ppitch);
            pk += 32u;
            up += --left == 0 ? sub - (uint32_t)(a.gsub - 1) * 32u : 32u;                      // the second box
          });
          if (!settled) { peer_wait(&bars.stat); __syncwarp(); settled = true; }
#pragma unroll
          for (int g = 0; g < MG; ++g) {
            const int k = p * a.pg + kp0 + g;
            if (g > 0 && kp0 + g >= cnt) break;
            const int own = (int)(((float)((k + 1) * C - 1) + 0.5f) * inv_ng), kl = k - (own * a.ng >> a.lc);
            const uint32_t bar = map_to_cta(smem_addr(&bars.w), (uint32_t)own);
            const uint32_t dst = map_to_cta(s_u + (uint32_t)(((rank * a.gs + kl) * 16 + gid) * RW + part * TN * 8 + 2 * t4) * 4u, (uint32_t)own);
#pragma unroll
            for (int t = 0; t < TN; ++t) {
              st_async_f32x2(dst + t * 32u, acc[g][t][0], acc[g][t][1], bar);
              st_async_f32x2(dst + 8u * RW * 4u + t * 32u, acc[g][t][2], acc[g][t][3], bar);
            }
          }
        }
        first -= tasks;
        release();
      }
      // vision maximum and sum of every head over blocks and column ranges
      if (!settled) { peer_wait(&bars.stat); __syncwarp(); }
      if (SPR_WARPS - 1 - warp < G) {                         // (the last warps have the fewest granules)
        const int g = SPR_WARPS - 1 - warp, cnt = Re << a.lc;
        float mx = -INFINITY, s = 0.f;
#pragma unroll 1
        for (int i = lane; i < cnt; i += 32) mx = fmaxf(mx, stat[(i & (C - 1)) * RP + (i >> a.lc) * G + g].x);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
#pragma unroll 1
        for (int i = lane; i < cnt; i += 32) { const float2 x = stat[(i & (C - 1)) * RP + (i >> a.lc) * G + g]; s = fmaf(x.y, fast_exp2(x.x - mx), s); }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) hstat[g] = make_float2(mx, s);
      }
    } else if (tid < G) {
      hstat[tid] = make_float2(-INFINITY, 0.f);
    }
    if (!EARLY_TEXT) text_part();
    named_barrier_sync(1, SPR_CONS);

    // ---------------- step 4: this CTA's value rows, relative to one reference maximum per head ----------------
    float ref[NH];                                            // of head gid (+ 8): over the vision logits and this CTA's text rows
    {
      float f[NH];
#pragma unroll
      for (int nh = 0; nh < NH; ++nh) {
        float mx = gid + 8 * nh < G ? hstat[gid + 8 * nh].x : -INFINITY;
#pragma unroll
        for (int w = 0; w < SPR_WARPS; ++w) mx = fmaxf(mx, tstat[w * 16 + gid + 8 * nh].x);
        ref[nh] = mx;
        f[nh] = m_run[nh] == -INFINITY ? 0.f : fast_exp2(m_run[nh] - mx);
      }
      scale_heads(f);
    }
    if (warp < G) {                                           // (reference maximum, text sum) of head `warp` to all CTAs
      const float2 t = tstat[(lane & 15) * 16 + warp];
      float mx = t.x, l;
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      mx = fmaxf(mx, hstat[warp].x);
      l = t.y * spread_weight(t.x, mx);
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
      if (lane < C) st_async_f32x2(map_to_cta(smem_addr(&ystat[rank * 16 + warp]), (uint32_t)lane), mx, l, map_to_cta(smem_addr(&bars.y), (uint32_t)lane));
    }
    if (Re > 0) {
      peer_wait(&bars.w);
      __syncwarp();
      int first = warp;
#pragma unroll 1
      for (int r0 = 0; r0 < Re; r0 += a.bpp)
#pragma unroll 1
        for (int x = 0; x < kp; ++x) {
          const uint32_t pc = smem_addr(acquire());
          const int cnt = min(a.kg, gown - x * a.kg), tasks = min(a.bpp, Re - r0) * cnt;
          const uint32_t inv = x + 1 < kp ? inv_full : inv_last;
#pragma unroll 1
          for (; first < tasks; first += SPR_WARPS) {
            const int bl = (int)((uint32_t)first * inv >> 16), gi = first - bl * cnt, r = r0 + bl;
            float w[NH][4];
#pragma unroll
            for (int nh = 0; nh < NH; ++nh) {
#pragma unroll
              for (int e = 0; e < 4; ++e) w[nh][e] = 0.f;
              const int row = r * G + gid + 8 * nh;
              if (gid + 8 * nh < G) {
                const float* wr = Wr + ((x * a.kg + gi) * 16 + 2 * t4) * RW + row;
                const float2* st = stat + row;
#pragma unroll 2
                for (int c = 0; c < C; ++c, wr += a.gs * 16 * RW, st += RP) {
                  const float f = fast_exp2(st->x - ref[nh]);
                  w[nh][0] = fmaf(f, wr[0], w[nh][0]); w[nh][1] = fmaf(f, wr[RW], w[nh][1]);
                  w[nh][2] = fmaf(f, wr[8 * RW], w[nh][2]); w[nh][3] = fmaf(f, wr[9 * RW], w[nh][3]);
                }
              }
            }
            const uint32_t half = (uint32_t)a.kg * 2048u;
            values16(pc + (uint32_t)bl * 2u * half + (uint32_t)gi * 2048u, half, w);
          }
          first -= tasks;
          release();
        }
    }
    // ---------------- the warps' outputs meet where weights, probabilities and pieces were, the CTAs' by ranges of channels ----------------
    named_barrier_sync(1, SPR_CONS);                          // all of them have been read, and nothing is on its way there
    float* yred = reinterpret_cast<float*>(sm + a.s_off);     // [SPR_WARPS][8][SPR_YLD]
    const int ld = 7 - a.lc, dc = 1 << ld;                    // channels of a CTA
    const int unit = fresh((int)blockIdx.x) >> a.lc, pair = a.nrg > 1 ? unit / a.nrg : unit, rg = unit - pair * a.nrg;      // (anew: kept until here they spill)
    const uint32_t ybar = smem_addr(&bars.y);
#pragma unroll
    for (int nh = 0; nh < NH; ++nh) {
      if (nh > 0) named_barrier_sync(1, SPR_CONS);
#pragma unroll
      for (int mt = 0; mt < 8; ++mt)
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (2 * t4 + (e & 1) + 8 * nh < G) yred[(warp * 8 + 2 * t4 + (e & 1)) * SPR_YLD + mt * 16 + gid + (e >> 1) * 8] = y[mt][nh][e];
      named_barrier_sync(1, SPR_CONS);
#pragma unroll 1
      for (int i = tid; i < min(8, G - 8 * nh) * 32; i += SPR_CONS) {
        const int gg = i >> 5, d0 = (i & 31) * 4;
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int w = 0; w < SPR_WARPS; ++w) {
          const float4 v = *reinterpret_cast<const float4*>(&yred[(w * 8 + gg) * SPR_YLD + d0]);
          s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
        }
        const int own = d0 >> ld;
        st_async_f32x4(map_to_cta(smem_addr(&yrecv[(rank * G + gg + 8 * nh) * dc + d0 - own * dc]), (uint32_t)own), s, map_to_cta(ybar, (uint32_t)own));
      }
    }
    __syncwarp();
    cluster_arrive();                                         // nothing is sent to a peer after this
    peer_wait(&bars.y);
    __syncwarp();
    spread_end<SPR_CONS>(a, C, G, ld, dc, tid, pair, unit, rg, rank, ystat, yrecv, hstat, mus, &rowmax[0], [] { named_barrier_sync(1, SPR_CONS); });
    if (dead) {
      if (lane == 0) atomicExch(a.status, (int)KVC_ERR_TIMEOUT);
      __nanosleep(50000);                                     // what a peer has sent and this CTA gave up on still lands in its memory
    }
    __syncwarp();
  }
  cluster_wait();
}

// ------------------------------------------------------------------------------------------ host side
constexpr size_t SPR_DYN_LIMIT = 231424;      // 227 KB less the barriers

// rows of theta as the tensor map addresses them: the copy made at layer creation, or the caller's own array
static const void* spread_theta(const kvc_layer* L) { return L->theta_rows ? L->theta_rows : L->desc.theta; }
static int spread_theta_np(const kvc_layer* L) { return L->theta_rows ? L->theta_np : L->desc.n; }

bool spread_may_serve(const kvc_layer* L) {
  return L->desc.dtype == KVC_BF16 && !L->passthrough && L->mode == KVC_MODE_KV && L->desc.n >= 64 && (L->use_tc == 0 || L->use_tc == 6);
}

// bf16 terms of the scores and probabilities: two where the general paths keep them in two or in fp32 (cluster_terms: n no multiple of 8, or more
// than some 720 retained rows), but one for the uniform calls of such long rows that the three-kernel or the one-kernel path takes, which
// carry one.  4 x 3 blocks of n = 1024, m = 820, 28/4 heads, with lengths per sequence, relative error of the output against 64 bits on peaked
// softmaxes: one term 3.9e-3, two 1.7e-3 (its rounding to bf16).
static int spread_terms(const kvc_layer* L, int B, int R, int T, bool ragged) {
  if (cluster_terms(L) == 1) return 1;
  const bool one = !ragged && L->desc.n % 64 == 0 && ((plan_split(L, B, R).ok && T <= 64 * SP_OUT_ROWS * SP_TEXT_CHUNK) || plan_fused(L, B, R).ok);
  return one ? 1 : 2;
}

// most_waves: 1: clusters for all groups at once; more: clusters of two, in that many waves at most
static SpreadPlan plan_groups(const kvc_layer* L, int B, int R_all, int T_all, int nrg, int most_waves, int terms) {
  SpreadPlan p{};
  const int R = ceil_div(R_all, nrg), T = ceil_div(T_all, nrg);
  const int G = L->G, n = L->desc.n, m = L->m, H = L->desc.H_kv;
  p.nrg = nrg; p.rg = R;
  if (R > 64 || R * G > 64 || (nrg - 1) * R >= R_all) return p;
  p.ng = ceil_div(m, 16);
  p.ncg = ceil_div(n, 16);
  for (int c = SPR_MAX_C; c >= 2; c /= 2)
    if ((long long)B * H * nrg <= L->clusters[c] && p.ng >= c && p.ncg >= c) { p.C = c; break; }
  p.waves = 1;
  if (p.C == 0 && most_waves > 1 && L->clusters[2] > 0 && p.ng >= 2 && p.ncg >= 2) {
    const long long w = ((long long)B * H * nrg + L->clusters[2] - 1) / L->clusters[2];
    if (w <= most_waves) { p.C = 2; p.waves = (int)w; }
  }
  if (p.C == 0) return p;
  p.gs = ceil_div(p.ng, p.C);
  p.gw = ceil_div(p.ncg, p.C);
  if (p.gw > SPR_WARPS) return p;
  p.nt = ceil_div(R * G, 8);
  if (p.nt > 1) p.nt = (p.nt + 1) & ~1;
  if (G > 8 && p.nt == 6) p.nt = 8;
  p.terms = terms;
  p.nsub = p.gw > 15 ? 2 : 1;
  p.gsub = ceil_div(p.gw, p.nsub);
  p.wbox = p.gsub * 16 + 8;
  const uint32_t gran = (uint32_t)(p.nsub * 16 * p.wbox) * 2u;
  const int RP = p.nt * 8;
  uint32_t off = 0;
  auto take = [&](uint32_t bytes) { const uint32_t o = off; off = (off + bytes + 127u) & ~127u; return o; };
  p.misc_off = take((uint32_t)(RP * 4 + SPR_WARPS * RP * 4 + SPR_MAX_C * RP * 8 + SPR_WARPS * 16 * 8 + 16 * 8 + SPR_MAX_C * 16 * 8 + D * 2));
  p.q_off = take(16u * SPR_QPITCH);
  p.y_off = take((uint32_t)(G * D * 4));
  const uint32_t S = (uint32_t)(p.C * p.terms * RP * (p.gs * 16 + 8) * 2), W = (uint32_t)(p.C * p.gs * 16 * (RP + 4) * 4);
  p.s_off = take(S > W ? S : W);
  p.p_off = take((uint32_t)(p.terms * RP * (p.gw * 16 + 8) * 2));
  p.ring_off = (off + 1023u) & ~1023u;
  if (p.ring_off + 1024u + 4u * 8192u >= SPR_DYN_LIMIT) return p;
  // A piece is looked at by every warp (about 200 cycles a look): few large ones, five of which fill the ring, four with a single row tile (1 x 5
  // blocks of n = 576, 32/32 heads: 12.8 us, five 13.2, seven 14.2; 2 x 4 of 1024, 32/8 heads, two tiles: 18.5, 17.5, 19.5)
  const uint32_t room = (uint32_t)SPR_DYN_LIMIT - 1024u - p.ring_off, want = room / (p.nt == 1 ? 4u : 5u) & ~1023u;
  const int kp = ceil_div(p.gs, 16);
  p.kg = ceil_div(p.gs, kp);
  p.bpp = std::max(1, std::min(kp > 1 ? 1 : R, (int)(want / ((uint32_t)p.kg * 4096u))));
  p.bpp = ceil_div(R, ceil_div(R, p.bpp));
  p.pg = std::max(1, std::min(std::min(16, p.ng), (int)(want / gran)));
  p.npp = ceil_div(p.ng, p.pg);
  p.pg = ceil_div(p.ng, p.npp);
  if (p.nt > 2) p.pg = std::min(16, (p.pg + 1) & ~1);          // granules are taken in pairs
  p.npp = ceil_div(p.ng, p.pg);
  p.ti = std::max(1, std::min(std::min(16, ceil_div(ceil_div(T, 16), p.C)), (int)(want / 8192u)));
  p.slot_bytes = std::max(std::max((uint32_t)(p.kg * p.bpp) * 4096u, gran * p.pg), (uint32_t)p.ti * 8192u);
  p.slot_bytes = (p.slot_bytes + 1023u) & ~1023u;
  p.slots = std::min((int)(room / p.slot_bytes), SPR_MAX_SLOTS);
  if (p.slots < 2 || p.ring_off - p.s_off + (uint32_t)p.slots * p.slot_bytes < SPR_WARPS * 8u * SPR_YLD * 4u) return p;
  p.smem = 1024u + (size_t)p.ring_off + (size_t)p.slots * p.slot_bytes;
  {
    // us of a call: the looks at pieces, the steps of the two expansions of a warp, its text items, the exchanged weights, the bytes.  Fitted
    // (non-negative least squares of the relative error, 6 %) to 260 calls on B200: 110 drawn shapes, every number of groups they allow
    const int items = ceil_div(ceil_div(T_all, 16), p.C * nrg), MG = p.nt > 2 ? 2 : 1, TN = p.nt > 2 ? p.nt / 2 : p.nt;
    int tasks = 0;
    for (int x = 0; x < p.npp; ++x) { const int c = std::min(p.pg, p.ng - x * p.pg); tasks += MG == 2 ? (c + 1) & ~1 : c; }
    const double step = TN * p.terms * MG, pieces = 2.0 * ceil_div(R, p.bpp) * kp + 2.0 * p.npp + ceil_div(items, p.ti);
    const double at_once = p.waves > 1 ? L->clusters[2] : (double)B * H * nrg;
    const double mb = (at_once * p.C * (2.0 * R * p.gs * 4096.0 + items * 8192.0) + 4.0 * H * n * (double)m) * 1e-6;
    p.us = 5.9 + (nrg > 1 ? 3.6 : 0.0) + 0.336 * pieces + 0.0292 * p.ng * step + 0.0086 * ceil_div(tasks, SPR_WARPS) * p.gw * step +
           0.45 * ceil_div(items, SPR_WARPS) + 0.0525 * W / 1024.0 + 0.0485 * mb;
    // two tiles of query heads: the values, the text and the ends take twice as long (881 calls of G = 9 to 16: 10 %, without this 1.5 times too short)
    if (G > 8) p.us = 1.106 * p.us - 0.96 + 0.298 * items + 5.23 * ceil_div(R * p.gs, SPR_WARPS);
    // (394 calls of 220 shapes, one to four waves: 6 %)
    if (p.waves > 1) p.us = 0.9 + p.waves * (0.63 + 0.86 * p.us);
  }
  p.ok = 1;
  return p;
}

// Groups of blocks per pair: as many as 64 expansion rows each demand, more where the estimate finds the shorter chain of a group worth the
// merge (us per call: 1 x 31 blocks of n = 576, m = 432, 16/2 heads, 4 groups 40.5, 6 30.1, 8 25.6, the one-kernel path 43.7; 4 x 5 of 1024,
// 28/4 heads, one 33.1, two 26.5; 1 x 5 of 576, 28/4 heads, one 15.6, two 16.8, three 15.0).  Of the 110 shapes above each takes 14.31 us (geometric
// mean) with its best number, 14.36 with the chosen one, 15.5 with the smallest, 23.8 on the paths below.
SpreadPlan plan_spread(const kvc_layer* L, int B, int R, int T, bool ragged) {
  if (!spread_may_serve(L) || B < 1 || R < 1 || L->G > 16 || T < 0) return SpreadPlan{};
  if (!tma_rows(spread_theta(L)) || !tma_rows(L->U_rows) || spread_theta_np(L) % 8 || L->U_np % 8) return SpreadPlan{};
  SpreadPlan best{};
  const int terms = spread_terms(L, B, R, T, ragged);
  for (int nrg = 1; nrg <= SPR_MAX_NRG && nrg <= R; ++nrg) {
    const SpreadPlan p = plan_groups(L, B, R, T, nrg, 1, terms);
    if (p.ok && (!best.ok || p.us < best.us)) best = p;
  }
  // more groups than clusters the device holds: beside the paths for block lengths off 64 only (the others are ahead of a second wave: 30 x 2
  // blocks of n = 576, 28/4 heads 43 / 21.5; 21 x 2 of 1024 79 / 70)
  for (int nrg = 1; !best.ok && L->desc.n % 64 != 0 && nrg <= SPR_MAX_NRG && nrg <= R; ++nrg) {
    const SpreadPlan p = plan_groups(L, B, R, T, nrg, SPR_MAX_WAVES, terms);
    if (p.ok) best = p;
  }
  return best;
}

SpreadWs spread_ws(const kvc_layer* L, const SpreadPlan& p, int B) {
  SpreadWs w{};
  const size_t pairs = (size_t)B * L->desc.H_kv, parts = p.ok && p.nrg > 1 ? pairs * p.nrg : 0;
  size_t off = align_up(sizeof(int) * (pairs + 1), 256);                // behind the status word of the layout all paths share
  auto take = [&](size_t bytes) { const size_t o = off; off = align_up(off + bytes, 256); return o; };
  w.off_cnt = take(parts ? sizeof(unsigned long long) * pairs * p.C : 0);
  w.off_py = take(sizeof(float) * parts * L->G * D);
  w.off_pml = take(sizeof(float2) * parts * p.C * L->G);
  w.bytes = off;
  return w;
}

// enough for every T and for lengths per sequence: the number of groups and of terms depends on them, whether a number of groups can be had only on the terms
size_t spread_ws_bytes(const kvc_layer* L, int B, int R) {
  size_t most = 0;
  if (!plan_spread(L, B, R, 0, false).ok && !plan_spread(L, B, R, 0, true).ok) return 0;
  for (int terms = 1; terms <= cluster_terms(L); ++terms)
    for (int nrg = 1; nrg <= SPR_MAX_NRG && nrg <= R; ++nrg) {
      const SpreadPlan p = plan_groups(L, B, R, 0, nrg, SPR_MAX_WAVES, terms);
      if (p.ok) most = std::max(most, spread_ws(L, p, B).bytes);
    }
  return most;
}

template <int NT, int NH, int PL>
static cudaError_t launch_spread_inst(const CUtensorMap* tm, const SpreadArgs& a, const SpreadPlan& p, cudaStream_t st) {
  const cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(spread_decode_kernel<NT, NH, PL>), SPR_DYN_LIMIT);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(a.B * a.H_kv * p.nrg * p.C));
  cfg.blockDim = dim3(SPR_THREADS);
  cfg.dynamicSmemBytes = p.smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)p.C; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, spread_decode_kernel<NT, NH, PL>, tm[0], tm[1], tm[2], tm[3], tm[4], tm[5], a);
}
template <int PL>
static cudaError_t launch_spread_nt(const CUtensorMap* tm, const SpreadArgs& a, const SpreadPlan& p, cudaStream_t st) {
  if (a.G > 8)
    return p.nt == 2 ? launch_spread_inst<2, 2, PL>(tm, a, p, st) : (p.nt == 4 ? launch_spread_inst<4, 2, PL>(tm, a, p, st) : launch_spread_inst<8, 2, PL>(tm, a, p, st));
  switch (p.nt) {
    case 1: return launch_spread_inst<1, 1, PL>(tm, a, p, st);
    case 2: return launch_spread_inst<2, 1, PL>(tm, a, p, st);
    case 4: return launch_spread_inst<4, 1, PL>(tm, a, p, st);
    case 6: return launch_spread_inst<6, 1, PL>(tm, a, p, st);
    default: return launch_spread_inst<8, 1, PL>(tm, a, p, st);
  }
}

cudaError_t launch_spread(const kvc_layer* L, const DecodeArgs& d, const SpreadPlan& p, char* ws, cudaStream_t st, bool* encoded) {
  *encoded = false;
  const int B = d.B, H = d.H_kv, R = d.R, m = L->m, n = L->desc.n;
  CUtensorMap tm[6];
  {
    // capsule rows as (64 channels, m rows of a block, channel half, blocks): a box lands as [block][half][rows][64]
    const uint64_t dims[4] = {64ull, (uint64_t)m, 2ull, (uint64_t)B * H * R};
    const uint64_t str[3] = {256ull, 128ull, (uint64_t)m * 256};
    const uint32_t box[4] = {64u, (uint32_t)(16 * p.kg), 2u, (uint32_t)p.bpp};
    if (!encode_tensor_map_bf16(&tm[0], d.Kc, 4, dims, str, box) || !encode_tensor_map_bf16(&tm[1], d.Vc, 4, dims, str, box)) return cudaSuccess;
  }
  if (d.T > 0) {
    const uint64_t dims[5] = {64ull, (uint64_t)d.T, 2ull, (uint64_t)H, (uint64_t)B};
    const uint64_t str[4] = {256ull, 128ull, (uint64_t)d.T_cap * 256, (uint64_t)H * d.T_cap * 256};
    const uint32_t box[5] = {64u, (uint32_t)(16 * p.ti), 2u, 1u, 1u};
    if (!encode_tensor_map_bf16(&tm[2], d.K_txt, 5, dims, str, box) || !encode_tensor_map_bf16(&tm[3], d.V_txt, 5, dims, str, box)) return cudaSuccess;
  } else {
    tm[2] = tm[0];
    tm[3] = tm[1];
  }
  for (int x = 0; x < 2; ++x) {
    // theta, U as (n columns, m rows, H_kv), not swizzled: the odd number of 16-byte units in a box's row keeps ldmatrix free of conflicts
    const int np = x == 0 ? spread_theta_np(L) : L->U_np;
    const uint64_t dims[3] = {(uint64_t)n, (uint64_t)m, (uint64_t)H};
    const uint64_t str[2] = {(uint64_t)np * 2, (uint64_t)m * np * 2};
    const uint32_t box[3] = {(uint32_t)p.wbox, (uint32_t)(16 * p.pg), 1u};
    if (!encode_tensor_map_bf16(&tm[4 + x], x == 0 ? spread_theta(L) : L->U_rows, 3, dims, str, box, false)) return cudaSuccess;
  }
  *encoded = true;
  SpreadArgs a{};
  a.q = static_cast<const __nv_bfloat16*>(d.q);
  a.mu = static_cast<const __nv_bfloat16*>(d.mu);
  a.out = static_cast<__nv_bfloat16*>(d.out);
  const SpreadWs w = spread_ws(L, p, B);
  a.cnt = reinterpret_cast<unsigned long long*>(ws + w.off_cnt);
  a.py = reinterpret_cast<float*>(ws + w.off_py);
  a.pml = reinterpret_cast<float2*>(ws + w.off_pml);
  a.token = d.token; a.nrg = p.nrg; a.rg = p.rg;
  a.status = d.status; a.R_b = d.R_b; a.T_b = d.T_b; a.early = d.early_capsules;
  a.B = B; a.H_kv = H; a.G = d.G; a.R = R; a.m = m; a.n = n; a.T = d.T;
  a.lc = p.C == 8 ? 3 : (p.C == 4 ? 2 : 1); a.ng = p.ng; a.gs = p.gs; a.ncg = p.ncg; a.gw = p.gw; a.nsub = p.nsub; a.gsub = p.gsub; a.wbox = p.wbox;
  a.pg = p.pg; a.npp = p.npp; a.kg = p.kg; a.bpp = p.bpp; a.ti = p.ti; a.slots = p.slots;
  a.slot_bytes = p.slot_bytes; a.misc_off = p.misc_off; a.q_off = p.q_off; a.y_off = p.y_off; a.s_off = p.s_off; a.p_off = p.p_off; a.ring_off = p.ring_off;
  ProfScope prof(KVC_KERNEL_FUSED, st, KVC_KERNEL_SPREAD);
  return p.terms == 1 ? launch_spread_nt<1>(tm, a, p, st) : launch_spread_nt<2>(tm, a, p, st);
}

}  // namespace kvc
