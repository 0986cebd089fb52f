// The spread decode path (kvc_spread.cuh) for fp32 storage: small calls, every product on the CUDA cores in fp32.
//
// A (sequence, KV head) and a group of its blocks (at most 16 expansion rows) is served by a cluster of C CTAs that share the retained rows and
// the n axis; slices of S, row statistics, partial weights and outputs go through distributed shared memory as on the bf16 path.
//   step 1   eight threads per key row (16 channels each), the queries in shared memory; S is kept [retained row][expansion row]
//   step 2   a thread per (column, part of the retained rows): theta straight from global memory, S broadcast; the parts are summed
//            through shared memory
//   step 3   a thread per retained row (two where they fit): its row of U in shared memory, P broadcast
//   step 4   a warp per value row, four channels per lane; text rows the same way with their weights in shared memory
// 1 x 1 block of n = 576, 8/2 heads, 32 text rows: 35.1 us (four launches) -> 13.6; 4 x 3 of 256, 28/4 heads, 3173 rows 123 -> 35; 1 x 16 of 576,
// m = 389, 8/2 heads 108 -> 31; 8 x 1 of 1024, m = 794 87 -> 81 (calls of a captured graph back to back).
// Error against 64 bits, 59 shapes, relative to the three-phase kernels': 0.81 with peaked softmaxes, 0.94 with flat ones (geometric means).
// Bound: the chain of these steps and of four exchanges; theta and U come at the rate of the SMs that take part.
#include <algorithm>

#include "kvc_spread_end.cuh"

namespace kvc {

constexpr int SPF_THREADS = 512, SPF_WARPS = 16;
constexpr float SPF_QSCALE = 0.08838834764831845f * 1.4426950408889634f;      // sigma = 1/sqrt(128), logits in log2 units
constexpr int SPF_MAX_TEXT = 512;             // text rows per CTA
constexpr int SPF_MAX_NRG = 64, SPF_MAX_WAVES = 4;      // groups of blocks per pair; waves of clusters
constexpr int SPF_AHEAD = 12;                 // loads of theta per thread ahead of the scores

struct SpreadF32Args {
  const float *q, *mu, *Kc, *Vc, *K_txt, *V_txt, *theta, *U;
  float* out;
  float* py;             // (see SpreadWs)
  float2* pml;
  unsigned long long* cnt;
  unsigned int token;
  int* status;
  const int* R_b;
  const int* T_b;
  int early;
  int B, H_kv, G, R, m, n, T, T_cap, nrg, rg;
  int lc, js, qw, jc, vec;      // log2 CTAs per cluster; most retained rows and column quads of a CTA; rows per chunk of U; U in 16-byte copies
  uint32_t misc_off, q_off, y_off, s_off, w_off, red_off, p_off, t_off, u_off, u_pitch;      // u_pitch: floats per row of U (an odd multiple of 4)
};

__device__ __forceinline__ void cp_async4(uint32_t dst, const void* src, bool ok) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(dst), "l"(src), "r"(ok ? 4 : 0) : "memory");
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, int bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

// RT: expansion rows (row r G + g), padded; GT: query heads, padded
template <int RT, int GT>
__global__ void __launch_bounds__(SPF_THREADS, 1) spread_f32_kernel(const __grid_constant__ SpreadF32Args a) {
  constexpr int RL = RT + 4;                  // pitch of a row of P and of the partial logits: 16-byte accesses of 8 threads hit 32 banks
  extern __shared__ __align__(128) unsigned char sm[];
  __shared__ __align__(8) uint64_t bar_s, bar_stat, bar_w, bar_y;
  __shared__ int s_last;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int C = 1 << a.lc, G = a.G, rank = (int)blockIdx.x & (C - 1), unit = (int)blockIdx.x >> a.lc;
  const int pair = unit / a.nrg, rg = unit - pair * a.nrg, b = pair / a.H_kv, h = pair - b * a.H_kv;
  const int m = a.m, n = a.n;
  const bool ragged = a.R_b != nullptr || a.T_b != nullptr;
  const int j0 = rank * m >> a.lc, jn = ((rank + 1) * m >> a.lc) - j0;          // this CTA's retained rows
  const int nq = (n + 3) >> 2, q0 = rank * nq >> a.lc, c0 = q0 * 4, W = min((((rank + 1) * nq >> a.lc) - q0) * 4, n - c0);      // and columns
  const int W4 = (W + 3) & ~3;

  float2* stat = reinterpret_cast<float2*>(sm + a.misc_off);                    // [C][RT] (maximum, sum), written by the peers
  float2* hstat = stat + SPR_MAX_C * RT;                                        // [16] vision (maximum, sum) per head
  float2* ystat = hstat + 16;                                                   // [C][16] (reference maximum, text sum), written by the peers
  float* tmax = reinterpret_cast<float*>(ystat + SPR_MAX_C * 16);               // [16] text maximum per head
  float* tsum = tmax + 16;                                                      // [16] text sum relative to the reference maximum
  float* mus = tsum + 16;                                                       // [128 / C]
  float* qs = reinterpret_cast<float*>(sm + a.q_off);                           // [G][128], scaled
  float* yrecv = reinterpret_cast<float*>(sm + a.y_off);                        // [C][G][128 / C], written by the peers
  float* S = reinterpret_cast<float*>(sm + a.s_off);                            // [m][RT]; then the partial weights [C][js][RT]
  float* Wc = reinterpret_cast<float*>(sm + a.w_off);                           // [js][RT] joined weights
  float* red = reinterpret_cast<float*>(sm + a.red_off);                        // [parts][W][RL] partial logits
  float* P = reinterpret_cast<float*>(sm + a.p_off);                            // [W4][RL]
  float* ts = reinterpret_cast<float*>(sm + a.t_off);                           // [text rows][GT]
  float* Us = reinterpret_cast<float*>(sm + a.u_off);                           // [2][jc][u_pitch]

  if (tid < 4) {
    uint64_t* bar = tid == 0 ? &bar_s : (tid == 1 ? &bar_stat : (tid == 2 ? &bar_w : &bar_y));
    mbar_init(bar, 1);
    fence_mbar_init();
    mbar_expect_tx(bar, tid == 0 ? (uint32_t)((m - jn) * RT * 4) : (tid == 1 ? (uint32_t)(C * RT * 8) :
                        (tid == 2 ? (uint32_t)(C * jn * RT * 4) : (uint32_t)(G * D * 4 + C * G * 8))));
  }
  // parameters may be read before the stream's previous kernel has finished: the first two chunks of U to shared memory, theta into L2
  const float* theta = a.theta + (size_t)h * m * n + c0;
  const float* U = a.U + (size_t)h * m * n + c0;
  auto load_U = [&](int k) {                                   // chunk k, rows [k jc, ...)
    const int rows = min(a.jc, m - k * a.jc);
    const uint32_t dst = smem_addr(Us + (size_t)(k & 1) * a.jc * a.u_pitch);
    if (a.vec) {
      const int per = W4 >> 2;
#pragma unroll 1
      for (int i = tid; i < rows * per; i += SPF_THREADS) {
        const int j = i / per, x = i - j * per;
        cp_async16(dst + (uint32_t)(j * (int)a.u_pitch + x * 4) * 4u, U + (size_t)(k * a.jc + j) * n + x * 4, min(16, (W - x * 4) * 4));
      }
    } else {
#pragma unroll 1
      for (int i = tid; i < rows * W4; i += SPF_THREADS) {
        const int j = i / W4, x = i - j * W4;
        cp_async4(dst + (uint32_t)(j * (int)a.u_pitch + x) * 4u, U + (size_t)(k * a.jc + j) * n + min(x, W - 1), x < W);
      }
    }
  };
  const int nch = (m + a.jc - 1) / a.jc;
  {
    const int lines = (W * 4 + 127) / 128 + 1;
#pragma unroll 1
    for (int i = tid; i < m * lines; i += SPF_THREADS) {
      const int j = i / lines, x = min((i - j * lines) * 32, W - 1);
      prefetch_l2(theta + (size_t)j * n + x);
    }
  }
  load_U(0);
  cp_async_commit();
  if (nch > 1) load_U(1);
  cp_async_commit();
  const size_t blk0 = (size_t)pair * a.R + rg * a.rg;          // first block of the group in the capsule store
  if (a.early) {
    const int blocks = min(max(a.R - rg * a.rg, 0), a.rg);
#pragma unroll 1
    for (int i = tid; i < blocks * jn * 4; i += SPF_THREADS) {
      const int r = i / (jn * 4), x = i - r * jn * 4;
      prefetch_l2(a.Kc + ((blk0 + r) * m + j0) * D + x * 32);
      prefetch_l2(a.Vc + ((blk0 + r) * m + j0) * D + x * 32);
    }
  }
  __syncthreads();
  cluster_arrive();
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
  bool dead = false;
  auto peer_wait = [&](uint64_t* bar) { if (!dead && !mbar_wait_cluster_bounded(bar, 0u)) dead = true; };
  int Re = a.R, Te = a.T;
  if (a.R_b) { const int r = a.R_b[b]; Re = r < 0 ? 0 : (r > a.R ? a.R : r); }
  if (a.T_b) { const int t = a.T_b[b]; Te = t < 0 ? 0 : (t > a.T ? a.T : t); }
  Re = min(max(Re - rg * a.rg, 0), a.rg);
  int t0, tn;                                                  // this CTA's text rows
  {
    const uint32_t c = (uint32_t)(rg * C + rank), parts = (uint32_t)a.nrg << a.lc, q = (uint32_t)Te / parts, rem = (uint32_t)Te - q * parts;
    t0 = (int)(c * q + min(c, rem)); tn = (int)(q + (c < rem ? 1u : 0u));
  }
  const float* Kt = a.K_txt + ((size_t)pair * a.T_cap + t0) * D;
  const float* Vt = a.V_txt + ((size_t)pair * a.T_cap + t0) * D;

#pragma unroll 1
  for (int i = tid; i < G * D; i += SPF_THREADS) qs[i] = a.q[(size_t)pair * G * D + i] * SPF_QSCALE;
  if (tid < D >> a.lc) mus[tid] = a.mu[h * D + rank * (D >> a.lc) + tid];
  __syncthreads();
  cluster_wait();                                              // the peers' barriers exist

  // one key row by eight threads (channels 4 l + 32 i .. + 3): the scores of all heads, in every one of them
  const int l8 = tid & 7;
  auto score_row = [&](const float* row, bool ok, float (&s)[GT]) {
    float4 x[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) x[i] = ok ? *reinterpret_cast<const float4*>(row + l8 * 4 + 32 * i) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int g = 0; g < GT; ++g) {
      s[g] = 0.f;
      if (g < G) {
        float part[4];                                           // (short chains, added as a tree: a score's error grows with the logits it makes)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float4 q = *reinterpret_cast<const float4*>(qs + g * D + l8 * 4 + 32 * i);
          part[i] = fmaf(q.w, x[i].w, fmaf(q.z, x[i].z, fmaf(q.y, x[i].y, q.x * x[i].x)));
        }
        s[g] = (part[0] + part[1]) + (part[2] + part[3]);
      }
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1)
#pragma unroll
      for (int g = 0; g < GT; ++g) s[g] += __shfl_xor_sync(0xffffffffu, s[g], o);
  };
  float th[SPF_AHEAD];
  const int KL = SPF_THREADS / W, kl = tid / W, col = tid - kl * W;             // step 2: part of the retained rows, column
  const bool mine = kl < KL;
  if (Re > 0) {
    // ---------------- step 1 ----------------
#pragma unroll 1
    for (int i0 = 0; i0 < Re * jn; i0 += SPF_THREADS / 8) {
      const int i = i0 + (tid >> 3), r = i / jn, j = i - r * jn;
      const bool ok = i < Re * jn;
      float s[GT];
      score_row(a.Kc + ((blk0 + (ok ? r : 0)) * m + j0 + (ok ? j : 0)) * D, ok, s);
#pragma unroll
      for (int g = 0; g < GT; ++g)
        if (ok && g < G && (g & 7) == l8) S[(j0 + j) * RT + r * G + g] = s[g];
    }
    fence_proxy_async();
    __syncthreads();
    if (warp == 0 && lane < C && lane != rank) {
      const uint32_t src = smem_addr(S + j0 * RT);
      bulk_s2peer(map_to_cta(src, (uint32_t)lane), src, (uint32_t)(jn * RT * 4), map_to_cta(smem_addr(&bar_s), (uint32_t)lane));
    }
#pragma unroll
    for (int e = 0; e < SPF_AHEAD; ++e) th[e] = mine && kl + e * KL < m ? __ldg(theta + (size_t)(kl + e * KL) * n + col) : 0.f;
  }
  // ---------------- text scores, while S travels ----------------
#pragma unroll 1
  for (int i0 = 0; i0 < tn; i0 += SPF_THREADS / 8) {
    const int t = i0 + (tid >> 3);
    float s[GT];
    score_row(Kt + (size_t)(t < tn ? t : 0) * D, t < tn, s);
#pragma unroll
    for (int g = 0; g < GT; ++g)
      if (t < tn && g < G && (g & 7) == l8) ts[t * GT + g] = s[g];
  }
  if (Re > 0) {
    // ---------------- step 2 ----------------
    peer_wait(&bar_s);
    float acc[RT];
#pragma unroll
    for (int k = 0; k < RT; ++k) acc[k] = 0.f;
    auto fma_rows = [&](float (&sum)[RT], const float* v, float x) {
#pragma unroll
      for (int k = 0; k < RT; k += 4) {
        const float4 s = *reinterpret_cast<const float4*>(v + k);
        sum[k] = fmaf(s.x, x, sum[k]); sum[k + 1] = fmaf(s.y, x, sum[k + 1]); sum[k + 2] = fmaf(s.z, x, sum[k + 2]); sum[k + 3] = fmaf(s.w, x, sum[k + 3]);
      }
    };
    if (mine) {
#pragma unroll
      for (int e = 0; e < SPF_AHEAD; ++e) if (kl + e * KL < m) fma_rows(acc, S + (kl + e * KL) * RT, th[e]);
#pragma unroll 1
      for (int j = kl + SPF_AHEAD * KL; j < m; j += 8 * KL) {
        float t[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) t[e] = j + e * KL < m ? __ldg(theta + (size_t)(j + e * KL) * n + col) : 0.f;
        // eight products at a time: in one chain over all of a thread's rows, where few threads share a column (n = 1024 on two CTAs: one), the
        // error was 1.7 times that of the three-phase kernels' four chains, now 0.7 (16 x 2 blocks of n = 900, 8/2 heads)
        float part[RT];
#pragma unroll
        for (int k = 0; k < RT; ++k) part[k] = 0.f;
#pragma unroll
        for (int e = 0; e < 8; ++e) if (j + e * KL < m) fma_rows(part, S + (j + e * KL) * RT, t[e]);
#pragma unroll
        for (int k = 0; k < RT; ++k) acc[k] += part[k];
      }
#pragma unroll
      for (int k = 0; k < RT; k += 4) *reinterpret_cast<float4*>(red + (size_t)tid * RL + k) = make_float4(acc[k], acc[k + 1], acc[k + 2], acc[k + 3]);
    }
    __syncthreads();
#pragma unroll 1
    for (int i = tid; i < W4 * (RT / 4); i += SPF_THREADS) {
      const int c = i / (RT / 4), k = (i - c * (RT / 4)) * 4;
      float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
      if (c < W)
        for (int p = 0; p < KL; p += 4) {
          float4 x[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) x[e] = p + e < KL ? *reinterpret_cast<const float4*>(red + (size_t)((p + e) * W + c) * RL + k) : make_float4(0.f, 0.f, 0.f, 0.f);
          s.x += (x[0].x + x[1].x) + (x[2].x + x[3].x); s.y += (x[0].y + x[1].y) + (x[2].y + x[3].y);
          s.z += (x[0].z + x[1].z) + (x[2].z + x[3].z); s.w += (x[0].w + x[1].w) + (x[2].w + x[3].w);
        }
      *reinterpret_cast<float4*>(P + c * RL + k) = s;
    }
    __syncthreads();
    if (warp < RT) {                                           // row `warp`: probabilities relative to its maximum over this CTA's columns
      float mx = -INFINITY, s = 0.f;
#pragma unroll 1
      for (int c = lane; c < W; c += 32) mx = fmaxf(mx, P[c * RL + warp]);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      mx = ceilf(mx);                                          // a whole number: the factors between CTAs, blocks and text are powers of two, exact
#pragma unroll 1
      for (int c = lane; c < W4; c += 32) {
        const float p = c < W ? fast_exp2(P[c * RL + warp] - mx) : 0.f;
        P[c * RL + warp] = p;
        s += p;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane < C) st_async_f32x2(map_to_cta(smem_addr(&stat[rank * RT + warp]), (uint32_t)lane), mx, s, map_to_cta(smem_addr(&bar_stat), (uint32_t)lane));
    }
  }
  // text maximum of every head
  __syncthreads();
  if (warp < G) {
    float mx = -INFINITY;
#pragma unroll 1
    for (int t = lane; t < tn; t += 32) mx = fmaxf(mx, ts[t * GT + warp]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (lane == 0) tmax[warp] = ceilf(mx);
  }
  if (Re > 0) {
    // ---------------- step 3 ----------------
    bool settled = false;                                      // all CTAs have read their S, whose memory the weights take
    const int halves = 2 * a.jc <= SPF_THREADS ? 2 : 1;         // threads per row of U
#pragma unroll 1
    for (int k = 0; k < nch; ++k) {
      cp_async_wait<1>();
      __syncthreads();
      const int rows = min(a.jc, m - k * a.jc);
      const float* Uk = Us + (size_t)(k & 1) * a.jc * a.u_pitch;
#pragma unroll 1
      for (int i = tid; i < ((rows * halves + 31) & ~31); i += SPF_THREADS) {
        const int jl = halves == 2 ? i >> 1 : i, part = halves == 2 ? i & 1 : 0, mid = ((W4 >> 2) + 1) >> 1;
        const int x0 = part ? mid * 4 : 0, x1 = halves == 2 && !part ? min(mid * 4, W4) : W4;
        const bool ok = jl < rows;
        float acc[RT];
#pragma unroll
        for (int e = 0; e < RT; ++e) acc[e] = 0.f;
        const float* u = Uk + (size_t)(ok ? jl : 0) * a.u_pitch;
#pragma unroll 2
        for (int x = x0; x < x1; x += 4) {
          const float4 uv = *reinterpret_cast<const float4*>(u + x);
          const float ux[4] = {uv.x, uv.y, uv.z, uv.w};
#pragma unroll
          for (int e = 0; e < 4; ++e)
#pragma unroll
            for (int y = 0; y < RT; y += 4) {
              const float4 p = *reinterpret_cast<const float4*>(P + (x + e) * RL + y);
              acc[y] = fmaf(p.x, ux[e], acc[y]); acc[y + 1] = fmaf(p.y, ux[e], acc[y + 1]);
              acc[y + 2] = fmaf(p.z, ux[e], acc[y + 2]); acc[y + 3] = fmaf(p.w, ux[e], acc[y + 3]);
            }
        }
        if (halves == 2)
#pragma unroll
          for (int e = 0; e < RT; ++e) acc[e] += __shfl_xor_sync(0xffffffffu, acc[e], 1);
        if (!settled) { peer_wait(&bar_stat); settled = true; }
        __syncwarp();
        if (ok && part == 0) {
          const int j = k * a.jc + jl, own = ((j + 1) * C - 1) / m, kl2 = j - (own * m >> a.lc);
          const uint32_t bar = map_to_cta(smem_addr(&bar_w), (uint32_t)own), dst = map_to_cta(smem_addr(S + (size_t)(rank * a.js + kl2) * RT), (uint32_t)own);
#pragma unroll
          for (int e = 0; e < RT; e += 4) st_async_f32x4(dst + e * 4u, make_float4(acc[e], acc[e + 1], acc[e + 2], acc[e + 3]), bar);
        }
      }
      __syncthreads();
      if (k + 2 < nch) load_U(k + 2);
      cp_async_commit();
    }
    if (!settled) peer_wait(&bar_stat);
    __syncwarp();
    if (SPF_WARPS - 1 - warp < G) {                            // vision maximum and sum of every head over blocks and column ranges
      const int g = SPF_WARPS - 1 - warp, cnt = Re << a.lc;
      float mx = -INFINITY, s = 0.f;
#pragma unroll 1
      for (int i = lane; i < cnt; i += 32) mx = fmaxf(mx, stat[(i & (C - 1)) * RT + (i >> a.lc) * G + g].x);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
#pragma unroll 1
      for (int i = lane; i < cnt; i += 32) { const float2 x = stat[(i & (C - 1)) * RT + (i >> a.lc) * G + g]; s = fmaf(x.y, fast_exp2(x.x - mx), s); }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane == 0) hstat[g] = make_float2(mx, s);
    }
  } else if (tid < G) {
    hstat[tid] = make_float2(-INFINITY, 0.f);
  }
  __syncthreads();
  // text weights relative to the reference maximum of the head (over the vision logits and this CTA's text rows), in place
  if (warp < G) {
    const float mx = fmaxf(hstat[warp].x, tmax[warp]);
    float s = 0.f;
#pragma unroll 1
    for (int t = lane; t < tn; t += 32) {
      const float p = spread_weight(ts[t * GT + warp], mx);
      ts[t * GT + warp] = p;
      s += p;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane < C) st_async_f32x2(map_to_cta(smem_addr(&ystat[rank * 16 + warp]), (uint32_t)lane), mx, s, map_to_cta(smem_addr(&bar_y), (uint32_t)lane));
  }
  if (Re > 0) {
    peer_wait(&bar_w);
    __syncwarp();
#pragma unroll 1
    for (int i = tid; i < jn * RT; i += SPF_THREADS) {
      const int jl = i / RT, row = i & (RT - 1), g = row % G;
      float w = 0.f;
      if (row < Re * G) {
        const float ref = fmaxf(hstat[g].x, tmax[g]);
#pragma unroll 2
        for (int c = 0; c < C; ++c) w = fmaf(fast_exp2(stat[c * RT + row].x - ref), S[(size_t)(c * a.js + jl) * RT + row], w);
      }
      Wc[jl * RT + row] = w;
    }
  }
  __syncthreads();
  // ---------------- step 4 and the text's values: a warp per row, channels 4 lane .. + 3 ----------------
  float4 y[GT];
#pragma unroll
  for (int g = 0; g < GT; ++g) y[g] = make_float4(0.f, 0.f, 0.f, 0.f);
  auto add_row = [&](const float4& v, const float* w) {
#pragma unroll
    for (int g = 0; g < GT; ++g)
      if (g < G) { const float x = w[g]; y[g].x = fmaf(x, v.x, y[g].x); y[g].y = fmaf(x, v.y, y[g].y); y[g].z = fmaf(x, v.z, y[g].z); y[g].w = fmaf(x, v.w, y[g].w); }
  };
#pragma unroll 1
  for (int i0 = warp; i0 < Re * jn; i0 += 4 * SPF_WARPS) {
    float4 v[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int i = i0 + e * SPF_WARPS, r = i / jn, j = i - r * jn;
      v[e] = i < Re * jn ? *reinterpret_cast<const float4*>(a.Vc + ((blk0 + r) * m + j0 + j) * D + lane * 4) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int i = i0 + e * SPF_WARPS, r = i / jn, j = i - r * jn;
      if (i < Re * jn) add_row(v[e], Wc + j * RT + r * G);
    }
  }
#pragma unroll 1
  for (int t = warp; t < tn; t += 4 * SPF_WARPS) {
    float4 v[4];
#pragma unroll
    for (int e = 0; e < 4; ++e)
      v[e] = t + e * SPF_WARPS < tn ? *reinterpret_cast<const float4*>(Vt + (size_t)(t + e * SPF_WARPS) * D + lane * 4) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int e = 0; e < 4; ++e) if (t + e * SPF_WARPS < tn) add_row(v[e], ts + (t + e * SPF_WARPS) * GT);
  }
  // ---------------- the warps' outputs meet where logits, probabilities and U were, the CTAs' by ranges of channels ----------------
  cp_async_wait<0>();                                          // (a group without blocks has not looked at its U)
  float* yred = red;                                           // [SPF_WARPS][8][SPR_YLD]
  const int ld = 7 - a.lc, dc = 1 << ld;
  const uint32_t ybar = smem_addr(&bar_y);
#pragma unroll
  for (int g0 = 0; g0 < GT; g0 += 8) {
    if (g0 > 0 && g0 >= G) break;
    __syncthreads();
#pragma unroll
    for (int g = 0; g < 8; ++g)
      if (g0 + g < GT && g0 + g < G) *reinterpret_cast<float4*>(yred + (warp * 8 + g) * SPR_YLD + lane * 4) = y[(g0 + g) % GT];
    __syncthreads();
    if (tid < min(8, G - g0) * 32) {
      const int gg = tid >> 5, d0 = (tid & 31) * 4;
      float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int w = 0; w < SPF_WARPS; ++w) {
        const float4 v = *reinterpret_cast<const float4*>(&yred[(w * 8 + gg) * SPR_YLD + d0]);
        s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
      }
      const int own = d0 >> ld;
      st_async_f32x4(map_to_cta(smem_addr(&yrecv[(rank * G + gg + g0) * dc + d0 - own * dc]), (uint32_t)own), s, map_to_cta(ybar, (uint32_t)own));
    }
  }
  __syncwarp();
  cluster_arrive();                                            // nothing is sent to a peer after this
  peer_wait(&bar_y);
  __syncwarp();
  spread_end<SPF_THREADS>(a, C, G, ld, dc, tid, pair, unit, rg, rank, ystat, yrecv, hstat, mus, &s_last, [] { __syncthreads(); });
  if (dead) {
    if (lane == 0) atomicExch(a.status, (int)KVC_ERR_TIMEOUT);
    __nanosleep(50000);                                        // what a peer has sent and this CTA gave up on still lands in its memory
  }
  __syncwarp();
  cluster_wait();
}

// ------------------------------------------------------------------------------------------ host side
constexpr size_t SPF_DYN_LIMIT = 231424;

bool spread_f32_may_serve(const kvc_layer* L) {
  return L->desc.dtype == KVC_F32 && !L->passthrough && L->mode == KVC_MODE_KV && (L->use_tc == 0 || L->use_tc == 6);
}

struct SpreadF32Layout { int js, qw, jc, rt, gt; uint32_t misc, q, y, s, w, red, p, t, u, pitch; };
static bool spread_f32_layout(const kvc_layer* L, int C, int nrg, int R, int T, SpreadF32Layout& o) {
  const int G = L->G, m = L->m, n = L->desc.n;
  o.rt = R * G <= 4 ? 4 : (R * G <= 8 ? 8 : 16);
  o.gt = G <= 4 ? 4 : (G <= 8 ? 8 : 16);
  o.js = ceil_div(m, C);
  o.qw = ceil_div(ceil_div(n, 4), C);
  const int W = o.qw * 4, KL = SPF_THREADS / W;
  if (KL < 1) return false;
  const int tn = ceil_div(T, C * nrg);
  if (tn > SPF_MAX_TEXT) return false;
  uint32_t off = 0;
  auto take = [&](size_t bytes) { const uint32_t x = off; off = (off + (uint32_t)bytes + 127u) & ~127u; return x; };
  o.misc = take(SPR_MAX_C * o.rt * 8 + 16 * 8 + SPR_MAX_C * 16 * 8 + 2 * 16 * 4 + D * 4);
  o.q = take((size_t)G * D * 4);
  o.y = take((size_t)G * D * 4);
  o.s = take((size_t)C * o.js * o.rt * 4);
  o.w = take((size_t)o.js * o.rt * 4);
  o.t = take((size_t)tn * o.gt * 4);
  o.red = take((size_t)SPF_THREADS * (o.rt + 4) * 4);
  o.p = take((size_t)W * (o.rt + 4) * 4);
  o.u = off;
  o.pitch = (uint32_t)(o.qw % 2 ? W : W + 4);
  const size_t row = (size_t)o.pitch * 4;
  if (off >= SPF_DYN_LIMIT || o.red + SPF_WARPS * 8u * SPR_YLD * 4u > SPF_DYN_LIMIT) return false;
  o.jc = (int)((SPF_DYN_LIMIT - off) / (2 * row));
  if (o.jc > ceil_div(m, 2)) o.jc = ceil_div(m, 2);
  // chunks of few rows leave the threads idle; the outputs of the warps take the memory from the partial logits on
  return o.jc >= 64 || o.jc >= ceil_div(m, 2);
}

// Groups of blocks of at most 16 expansion rows and the size of their clusters, by an estimate of the call: waves of clusters, the fused multiply-adds
// of a thread in the two expansions, rounds of key and value rows, the bytes of the parameters and of the call.  Fitted (non-negative least squares
// of the relative error, 7 %) to 281 calls on B200: 70 drawn shapes, one to four waves.  Their best choices take 52.0 us in the geometric
// mean, the chosen ones 52.8, the three-phase kernels 93.1.
SpreadPlan plan_spread_f32(const kvc_layer* L, int B, int R, int T) {
  SpreadPlan p{};
  if (!spread_f32_may_serve(L) || B < 1 || R < 1 || T < 0 || L->m < 8) return p;
  const int H = L->desc.H_kv, G = L->G, n = L->desc.n, m = L->m;
  for (int rg = std::min(16 / G, R), last = 0; rg >= 1; --rg) {
    const int nrg = ceil_div(R, rg), rows = ceil_div(R, nrg) * G;
    if (nrg == last || nrg > SPF_MAX_NRG) continue;
    last = nrg;
    for (int c = SPR_MAX_C; c >= 2; c /= 2) {
      SpreadF32Layout o{};
      if (L->clusters[c] < 1 || ceil_div(n, 4) < c || !spread_f32_layout(L, c, nrg, rows / G, T, o)) continue;
      const long long clusters = (long long)B * H * nrg, waves = (clusters + L->clusters[c] - 1) / L->clusters[c];
      if (waves > SPF_MAX_WAVES) continue;
      const int W = o.qw * 4, tn = ceil_div(T, c * nrg), rb = rows / G;
      const double chain = ceil_div(m, SPF_THREADS / W) * (double)o.rt, two = m <= SPF_THREADS ? 2.0 : 1.0;
      const double expand = 9.06e-3 * chain + 0.48e-3 * ceil_div((int)(m * two), SPF_THREADS) * W * o.rt / two;
      const double rounds = o.gt * (0.269 * (ceil_div(rb * o.js, 64) + ceil_div(tn, 64)) + 0.0175 * (ceil_div(rb * o.js, 16) + ceil_div(tn, 16)));
      const double act = (double)std::min(clusters, (long long)L->clusters[c]) * c, kb = m * (double)W * 8.0 / 1024.0;
      const double us = (nrg > 1 ? 2.8 : 0.0) + waves * (8.5 + expand + rounds + 0.0328 * kb + 0.0736 * 1e-6 * act * (m * (double)W * 8.0 + 2.0 * rb * o.js * 512.0 + tn * 1024.0));
      if (!p.ok || us < p.us) { p.ok = 1; p.nrg = nrg; p.rg = rb; p.C = c; p.us = us; p.waves = (int)waves; }
    }
  }
  return p;
}

// enough for every T (the number of groups depends on it)
size_t spread_f32_ws_bytes(const kvc_layer* L, int B, int R) {
  if (!spread_f32_may_serve(L) || B < 1 || R < 1 || (long long)B * L->desc.H_kv > (long long)SPF_MAX_WAVES * L->clusters[2]) return 0;
  SpreadPlan p{};
  p.ok = 1; p.C = SPR_MAX_C; p.nrg = (int)std::min<long long>(std::min(SPF_MAX_NRG, R), (long long)SPF_MAX_WAVES * L->clusters[2] / ((long long)B * L->desc.H_kv));
  return spread_ws(L, p, B).bytes;
}

template <int RT, int GT>
static cudaError_t launch_spread_f32_inst(const SpreadF32Args& a, size_t smem, cudaStream_t st) {
  const cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(spread_f32_kernel<RT, GT>), SPF_DYN_LIMIT);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((a.B * a.H_kv * a.nrg) << a.lc));
  cfg.blockDim = dim3(SPF_THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = 1u << a.lc; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, spread_f32_kernel<RT, GT>, a);
}

cudaError_t launch_spread_f32(const kvc_layer* L, const DecodeArgs& d, const SpreadPlan& p, char* ws, cudaStream_t st) {
  SpreadF32Layout o{};
  if (!spread_f32_layout(L, p.C, p.nrg, p.rg, d.T, o)) return cudaErrorInvalidConfiguration;
  const SpreadWs w = spread_ws(L, p, d.B);
  SpreadF32Args a{};
  a.q = static_cast<const float*>(d.q); a.mu = static_cast<const float*>(d.mu);
  a.Kc = static_cast<const float*>(d.Kc); a.Vc = static_cast<const float*>(d.Vc);
  a.K_txt = static_cast<const float*>(d.K_txt); a.V_txt = static_cast<const float*>(d.V_txt);
  a.theta = static_cast<const float*>(d.theta); a.U = static_cast<const float*>(d.U);
  a.out = static_cast<float*>(d.out);
  a.cnt = reinterpret_cast<unsigned long long*>(ws + w.off_cnt);
  a.py = reinterpret_cast<float*>(ws + w.off_py);
  a.pml = reinterpret_cast<float2*>(ws + w.off_pml);
  a.token = d.token; a.status = d.status; a.R_b = d.R_b; a.T_b = d.T_b; a.early = d.early_capsules;
  a.B = d.B; a.H_kv = d.H_kv; a.G = d.G; a.R = d.R; a.m = L->m; a.n = L->desc.n; a.T = d.T; a.T_cap = d.T_cap; a.nrg = p.nrg; a.rg = p.rg;
  a.lc = p.C == 8 ? 3 : (p.C == 4 ? 2 : 1); a.js = o.js; a.qw = o.qw; a.jc = o.jc;
  a.vec = a.n % 4 == 0 && (reinterpret_cast<uintptr_t>(d.U) & 15) == 0;
  a.misc_off = o.misc; a.q_off = o.q; a.y_off = o.y; a.s_off = o.s; a.w_off = o.w; a.red_off = o.red; a.p_off = o.p; a.t_off = o.t; a.u_off = o.u;
  a.u_pitch = o.pitch;
  size_t smem = o.u + (size_t)2 * o.jc * o.pitch * 4;
  const size_t need = o.red + (size_t)SPF_WARPS * 8 * SPR_YLD * 4;       // the warps' outputs
  if (smem < need) smem = need;
  ProfScope prof(KVC_KERNEL_FUSED, st, KVC_KERNEL_SPREAD);
#define KVC_SPF(RT) (o.gt == 4 ? launch_spread_f32_inst<RT, 4>(a, smem, st) : (o.gt == 8 ? launch_spread_f32_inst<RT, 8>(a, smem, st) : launch_spread_f32_inst<RT, 16>(a, smem, st)))
  if (o.rt == 4) return launch_spread_f32_inst<4, 4>(a, smem, st);
  if (o.rt == 8) return o.gt == 4 ? launch_spread_f32_inst<8, 4>(a, smem, st) : launch_spread_f32_inst<8, 8>(a, smem, st);
  return KVC_SPF(16);
#undef KVC_SPF
}

}  // namespace kvc
