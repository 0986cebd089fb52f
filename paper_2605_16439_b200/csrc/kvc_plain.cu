// Plain decode attention (see kvc_plain.cuh): out = softmax(sigma q K^T) V over uncompressed rows, flash-style.
//
// Bound: HBM.  Every CTA streams an equal run of the flat list of steps.  Inside a CTA every warp walks its own steps from its own ring of
// 4 KB pieces (K and V in turn), issuing its own copies and carrying (max, sum, y) per query head in registers: no barrier until the
// CTA's part of a pair ends, and the copies of the next part are already in flight then.  Twelve warps with four pieces (192 KB a SM) cover
// the round trip to HBM: 64 CTAs already draw 5.6 TB/s.
// Measured on B200 (us per call, before: the text-only mode of the one-kernel path, equal slices per pair through CTA-wide stages):
// 16 x 8704 rows, 28/4 heads 72 -> 52 (285 MB, 5.5 TB/s); 8 x 8448 38 -> 29; 32 x 2304 75 -> 29; 8 x 3000, 32/32 heads 89 -> 63;
// 64 x 33000 642 -> 640; 1 x 2304 12.1 -> 10.3; 1 x 33000 27.5 -> 20.
#include "kvc_fused.cuh"
#include "kvc_plain.cuh"
#include "kvc_split.cuh"

namespace kvc {

constexpr float PN_QSCALE = 0.08838834764831845f * 1.4426950408889634f;      // sigma = 1/sqrt(128), logits in log2 units
constexpr int PN_THREADS = PN_WARPS * 32;
constexpr int PN_HALF = PN_WARPS / 2;

template <int NH, int SLOTS>
__global__ void __launch_bounds__(PN_THREADS, 1)
plain_decode_kernel(const __grid_constant__ CUtensorMap tmKa, const __grid_constant__ CUtensorMap tmVa,
                    const __grid_constant__ CUtensorMap tmKb, const __grid_constant__ CUtensorMap tmVb, const PlainArgs a) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* sm = smem_raw + ((1024u - (smem_addr(smem_raw) & 1023u)) & 1023u);
  __shared__ __align__(8) uint64_t full_bar[PN_WARPS][SLOTS];
  __shared__ float s_max[PN_WARPS][16], s_sum[PN_WARPS][16];
  __shared__ int s_last;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int gid = lane >> 2, t4 = lane & 3;
  const int l7 = lane & 7, lmid = (lane >> 3) & 1, lrowB = l7 + (lane >> 4) * 8;
  const int G = a.G, spp = a.spp;
  float* red = reinterpret_cast<float*>(sm + a.off_red);                      // [PN_HALF][G][D]
  if (lane == 0) {
    for (int s = 0; s < SLOTS; ++s) mbar_init(&full_bar[warp][s], 1);
    fence_mbar_init();
  }
  __syncwarp();
  const long long lo = run_begin(blockIdx.x, a.total, gridDim.x), hi = run_begin(blockIdx.x + 1, a.total, gridDim.x);
  const int p_lo = (int)(lo / spp), p_hi = (int)((hi - 1) / spp);
  // this warp's steps of pair p: [w0, w1)
  auto share = [&](int p, int& w0, int& w1) {
    const long long base = (long long)p * spp;
    const int s0 = lo > base ? (int)(lo - base) : 0, s1 = hi < base + spp ? (int)(hi - base) : spp;
    w0 = s0 + (int)((long long)(s1 - s0) * warp / PN_WARPS);
    w1 = s0 + (int)((long long)(s1 - s0) * (warp + 1) / PN_WARPS);
  };
  unsigned char* ring = sm + (uint32_t)warp * (SLOTS * PN_PIECE);
  const uint32_t ring_u = smem_addr(ring);
  // ---- the copies of this warp, in the order it takes them
  int ip = p_lo, is = 0, ie = 0, iss = 0;
  bool ival = false;
  share(ip, is, ie);
  auto issue_next = [&]() {
    while (is >= ie) {
      if (ip >= p_hi) return;
      ++ip;
      share(ip, is, ie);
    }
    if (lane == 0) {
      const bool vis = is < a.steps_a;
      mbar_expect_tx(&full_bar[warp][iss], PN_PIECE);
      tma_load_4d(ring + iss * PN_PIECE, vis ? (ival ? &tmVa : &tmKa) : (ival ? &tmVb : &tmKb), 0, (vis ? is : is - a.steps_a) * PN_ROWS, 0, ip,
                  &full_bar[warp][iss]);
    }
    iss = iss + 1 < SLOTS ? iss + 1 : 0;
    if (ival) ++is;
    ival = !ival;
  };
  if (lane == 0) {
    tma_prefetch_desc(&tmKb); tma_prefetch_desc(&tmVb);
    if (a.steps_a > 0) { tma_prefetch_desc(&tmKa); tma_prefetch_desc(&tmVa); }
  }
  grid_dep_wait();
  grid_dep_launch();
  if (blockIdx.x == 0 && tid == 0) *a.status = 0;
#pragma unroll
  for (int x = 0; x < SLOTS; ++x) issue_next();

  int uss = 0;                                    // slot of the next piece taken, and the rounds' parities
  uint32_t pbits = 0;
  bool dead = false;
  auto wait_piece = [&]() {
    if (!dead && !mbar_wait_bounded(&full_bar[warp][uss], (pbits >> uss) & 1u)) dead = true;
    __syncwarp();
    pbits ^= 1u << uss;
    const uint32_t at = ring_u + (uint32_t)uss * PN_PIECE;
    uss = uss + 1 < SLOTS ? uss + 1 : 0;
    return at;
  };

  for (int p = p_lo; p <= p_hi; ++p) {
    int w0, w1;
    share(p, w0, w1);
    // A fragments of the logit product: rows = the heads of the group (gid, gid + 8), k = the 128 channels
    uint32_t qa[8][4];
    {
      const __nv_bfloat16* q0 = a.q + (size_t)p * G * D;
#pragma unroll
      for (int ks = 0; ks < 8; ++ks) {
        const int k0 = ks * 16 + 2 * t4;
        qa[ks][0] = gid < G ? *reinterpret_cast<const uint32_t*>(q0 + (size_t)gid * D + k0) : 0u;
        qa[ks][2] = gid < G ? *reinterpret_cast<const uint32_t*>(q0 + (size_t)gid * D + k0 + 8) : 0u;
        qa[ks][1] = NH > 1 && gid + 8 < G ? *reinterpret_cast<const uint32_t*>(q0 + (size_t)(gid + 8) * D + k0) : 0u;
        qa[ks][3] = NH > 1 && gid + 8 < G ? *reinterpret_cast<const uint32_t*>(q0 + (size_t)(gid + 8) * D + k0 + 8) : 0u;
      }
    }
    float yacc[8][NH][4];
#pragma unroll
    for (int mt = 0; mt < 8; ++mt)
#pragma unroll
      for (int nh = 0; nh < NH; ++nh)
#pragma unroll
        for (int e = 0; e < 4; ++e) yacc[mt][nh][e] = 0.f;
    float m_run[NH], l_run[NH];
#pragma unroll
    for (int nh = 0; nh < NH; ++nh) { m_run[nh] = -INFINITY; l_run[nh] = 0.f; }
    for (int s = w0; s < w1; ++s) {
      const int nv = s < a.steps_a ? a.S0 - s * PN_ROWS : a.T - (s - a.steps_a) * PN_ROWS;      // valid rows of the step (may exceed 16)
      // ---- keys: logits [16 heads][16 rows], two accumulation chains per 8-row group
      const uint32_t k_u = wait_piece() + (uint32_t)lrowB * 128u;
      float cc[2][4];
      {
        float c2[2][2][4];
#pragma unroll
        for (int x = 0; x < 2; ++x)
#pragma unroll
          for (int nt = 0; nt < 2; ++nt)
#pragma unroll
            for (int e = 0; e < 4; ++e) c2[x][nt][e] = 0.f;
#pragma unroll
        for (int ks = 0; ks < 8; ++ks) {
          uint32_t bk[4];
          ldsm_x4(bk, k_u + (ks >> 2) * 2048u + (uint32_t)(((((ks & 3) * 2 + lmid)) ^ l7) << 4));
          mma_bf16_16816(c2[ks & 1][0], qa[ks], bk[0], bk[1]);
          mma_bf16_16816(c2[ks & 1][1], qa[ks], bk[2], bk[3]);
        }
#pragma unroll
        for (int nt = 0; nt < 2; ++nt)
#pragma unroll
          for (int e = 0; e < 4; ++e) cc[nt][e] = (c2[0][nt][e] + c2[1][nt][e]) * PN_QSCALE;
      }
      __syncwarp();
      issue_next();
      // cc[nt][e]: head gid + 8 (e >> 1), row 8 nt + 2 t4 + (e & 1)
      if (nv < PN_ROWS) {
#pragma unroll
        for (int nt = 0; nt < 2; ++nt)
#pragma unroll
          for (int e = 0; e < 4; ++e)
            if (nt * 8 + 2 * t4 + (e & 1) >= nv) cc[nt][e] = -INFINITY;
      }
      float scl[NH];
#pragma unroll
      for (int hr = 0; hr < NH; ++hr) {
        float mx = fmaxf(fmaxf(cc[0][2 * hr], cc[0][2 * hr + 1]), fmaxf(cc[1][2 * hr], cc[1][2 * hr + 1]));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
        const float m_new = fmaxf(m_run[hr], mx);              // finite: a step holds at least one valid row
        scl[hr] = fast_exp2(m_run[hr] - m_new);
        m_run[hr] = m_new;
        float ps = 0.f;
#pragma unroll
        for (int nt = 0; nt < 2; ++nt)
#pragma unroll
          for (int x = 0; x < 2; ++x) {
            const float e = fast_exp2(cc[nt][2 * hr + x] - m_new);
            cc[nt][2 * hr + x] = e;
            ps += e;
          }
        l_run[hr] = l_run[hr] * scl[hr] + ps;
      }
#pragma unroll
      for (int nh = 0; nh < NH; ++nh) {
        if (__any_sync(0xffffffffu, scl[nh] != 1.f)) {
          const float c0s = __shfl_sync(0xffffffffu, scl[nh], (2 * t4) * 4);
          const float c1s = __shfl_sync(0xffffffffu, scl[nh], (2 * t4 + 1) * 4);
#pragma unroll
          for (int mt = 0; mt < 8; ++mt) {
            yacc[mt][nh][0] *= c0s; yacc[mt][nh][1] *= c1s;
            yacc[mt][nh][2] *= c0s; yacc[mt][nh][3] *= c1s;
          }
        }
      }
      // ---- values (rows past the last are zero-filled by the copy): y^T[128][heads] += V^T P^T
      uint32_t pb[NH][2];
#pragma unroll
      for (int nh = 0; nh < NH; ++nh) { pb[nh][0] = pack2_bf16(cc[0][2 * nh], cc[0][2 * nh + 1]); pb[nh][1] = pack2_bf16(cc[1][2 * nh], cc[1][2 * nh + 1]); }
      const uint32_t v_u = wait_piece() + (uint32_t)lrowB * 128u;
#pragma unroll
      for (int mt = 0; mt < 8; ++mt) {
        uint32_t av[4];
        ldsm_x4_t(av, v_u + (mt >> 2) * 2048u + (uint32_t)(((((mt & 3) * 2 + lmid)) ^ l7) << 4));
#pragma unroll
        for (int nh = 0; nh < NH; ++nh) mma_bf16_16816(yacc[mt][nh], av, pb[nh][0], pb[nh][1]);
      }
      __syncwarp();
      issue_next();
    }

    // ---------------- the CTA's part of the pair: the warps' states meet at one maximum per head ----------------
    if (t4 == 0) {
#pragma unroll
      for (int nh = 0; nh < NH; ++nh) s_max[warp][gid + 8 * nh] = m_run[nh];
    }
    __syncthreads();
    float M[NH];
    {
#pragma unroll
      for (int nh = 0; nh < NH; ++nh) {
        M[nh] = -INFINITY;
#pragma unroll
        for (int w = 0; w < PN_WARPS; ++w) M[nh] = fmaxf(M[nh], s_max[w][gid + 8 * nh]);
        const float sc = m_run[nh] == -INFINITY ? 0.f : fast_exp2(m_run[nh] - M[nh]);
        float l = l_run[nh] * sc;
        l += __shfl_xor_sync(0xffffffffu, l, 1);
        l += __shfl_xor_sync(0xffffffffu, l, 2);
        if (t4 == 0) s_sum[warp][gid + 8 * nh] = dead ? 0.f : l;
        const float c0s = __shfl_sync(0xffffffffu, sc, (2 * t4) * 4);
        const float c1s = __shfl_sync(0xffffffffu, sc, (2 * t4 + 1) * 4);
#pragma unroll
        for (int mt = 0; mt < 8; ++mt) {
          yacc[mt][nh][0] *= c0s; yacc[mt][nh][1] *= c1s;
          yacc[mt][nh][2] *= c0s; yacc[mt][nh][3] *= c1s;
        }
      }
    }
    // the upper half of the warps parks its accumulators, the lower half adds them to its own and parks the sums
#pragma unroll
    for (int round = 0; round < 2; ++round) {
      if ((warp >= PN_HALF) == (round == 0)) {
        float* mine = red + (size_t)(warp % PN_HALF) * (G * D);
#pragma unroll
        for (int nh = 0; nh < NH; ++nh)
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const int head = nh * 8 + 2 * t4 + e;
            if (head < G) {
              float* yp = mine + head * D;
#pragma unroll
              for (int mt = 0; mt < 8; ++mt) {
                if (round == 1) { yacc[mt][nh][e] += yp[mt * 16 + gid]; yacc[mt][nh][2 + e] += yp[mt * 16 + gid + 8]; }
                yp[mt * 16 + gid] = yacc[mt][nh][e];
                yp[mt * 16 + gid + 8] = yacc[mt][nh][2 + e];
              }
            }
          }
      }
      __syncthreads();
    }
    const int first = run_owner((long long)p * spp, a.total, gridDim.x), parts = run_owner((long long)(p + 1) * spp - 1, a.total, gridDim.x) - first + 1;
    const size_t slot = (size_t)p * a.slots + (blockIdx.x - first);
    for (int idx = tid; idx < G * (D / 4); idx += PN_THREADS) {
      const int head = idx >> 5, c = (idx & 31) * 4;
      float4 y = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int w = 0; w < PN_HALF; ++w) {
        const float4 v = *reinterpret_cast<const float4*>(red + (size_t)w * (G * D) + head * D + c);
        y.x += v.x; y.y += v.y; y.z += v.z; y.w += v.w;
      }
      float l = 0.f;
#pragma unroll
      for (int w = 0; w < PN_WARPS; ++w) l += s_sum[w][head];
      if (parts == 1) {
        const float inv = l > 0.f ? 1.f / l : 0.f;
        uint2 o;
        o.x = pack2_bf16(y.x * inv, y.y * inv); o.y = pack2_bf16(y.z * inv, y.w * inv);
        *reinterpret_cast<uint2*>(a.out + ((size_t)p * G + head) * D + c) = o;
      } else {
        *reinterpret_cast<float4*>(a.py + (slot * G + head) * D + c) = y;
        if (c == 0) {
          float m = -INFINITY;
#pragma unroll
          for (int w = 0; w < PN_WARPS; ++w) m = fmaxf(m, s_max[w][head]);
          a.pml[slot * G + head] = make_float2(m, l);
        }
      }
    }
    __syncthreads();                              // the partial is written; red and the statistics are free
    if (parts == 1) continue;
    if (tid == 0) {
      __threadfence();
      s_last = arrive_is_last(&a.cnt[p], a.token, parts) ? 1 : 0;
      __threadfence();
    }
    __syncthreads();
    if (s_last) {
      // lane <-> partial for the statistics, the values eight partials at a time
      for (int head = warp; head < G; head += PN_WARPS) {
        const size_t base = (size_t)p * a.slots;
        float2 st[2];
#pragma unroll
        for (int x = 0; x < 2; ++x) st[x] = lane + 32 * x < parts ? __ldcg(&a.pml[(base + lane + 32 * x) * G + head]) : make_float2(-INFINITY, 0.f);
        float mx = fmaxf(st[0].x, st[1].x);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        float f[2], den = 0.f;
#pragma unroll
        for (int x = 0; x < 2; ++x) { f[x] = st[x].x == -INFINITY ? 0.f : fast_exp2(st[x].x - mx); den = fmaf(f[x], st[x].y, den); }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) den += __shfl_xor_sync(0xffffffffu, den, o);
        float4 num = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int q = 0; q < parts; q += 8) {
          float4 y[8];
#pragma unroll
          for (int x = 0; x < 8; ++x)
            if (q + x < parts) y[x] = __ldcg(reinterpret_cast<const float4*>(a.py + ((base + q + x) * G + head) * D + lane * 4));
#pragma unroll
          for (int x = 0; x < 8; ++x) {
            const float w = __shfl_sync(0xffffffffu, q < 32 ? f[0] : f[1], (q + x) & 31);
            if (q + x < parts) { num.x = fmaf(w, y[x].x, num.x); num.y = fmaf(w, y[x].y, num.y); num.z = fmaf(w, y[x].z, num.z); num.w = fmaf(w, y[x].w, num.w); }
          }
        }
        const float inv = den > 0.f ? 1.f / den : 0.f;
        uint2 o;
        o.x = pack2_bf16(num.x * inv, num.y * inv); o.y = pack2_bf16(num.z * inv, num.w * inv);
        *reinterpret_cast<uint2*>(a.out + ((size_t)p * G + head) * D + lane * 4) = o;
      }
    }
  }
  if (dead && lane == 0) atomicExch(a.status, (int)KVC_ERR_TIMEOUT);
}

// ------------------------------------------------------------------------------------------ host side
// partial slots of a pair: CTAs that can share it (pair-aligned runs of at most sms / pairs CTAs, or crossing runs on all SMs)
static int part_slots(const kvc_layer* L, int B) {
  const long long n = (L->num_sms > 0 ? L->num_sms : 148) / ((long long)B * L->desc.H_kv) + 2;
  return (int)(n < PN_MAX_PARTS ? n : PN_MAX_PARTS);
}

PlainPlan plan_plain(const kvc_layer* L, int B, int S0, int T) {
  PlainPlan p{};
  const int G = L->G, H = L->desc.H_kv;
  if (L->desc.dtype != KVC_BF16 || B < 1 || S0 + T < 1 || G > 16) return p;
  if ((long long)B * H >= (1ll << 30)) return p;
  const int sms = L->num_sms > 0 ? L->num_sms : 148;
  p.steps_a = ceil_div(S0, PN_ROWS);
  p.spp = p.steps_a + ceil_div(T, PN_ROWS);
  p.total = (long long)B * H * p.spp;
  // CTAs: equal runs of the list whose ends fall on pair boundaries wherever possible, since a run that crosses one pays the end of a
  // pair twice.  Up to one pair per SM: as many CTAs per pair as the SMs allow, with at least 16 steps each (64 pairs x 544 steps: 128 CTAs
  // 51.5 us, 148 crossing 54; 32 x 528: 128 CTAs 29.3, 148 crossing 34), one where a pair has few steps (4 pairs x 44 steps: one CTA
  // each 8.6 us, 4 to 37 each 9.1 to 10.7).  More pairs than SMs: a CTA per pair (256 pairs x 7 steps 8.5 us, 148 crossing 14.8; x 188: 63.3 and
  // 67.2), unless the last wave of long pairs would be nearly empty: then equal runs on all SMs.
  const long long bh = (long long)B * H;
  long long grid;
  if (bh <= sms) {
    long long cpb = sms / bh, most = p.spp <= 48 ? 1 : ceil_div(p.spp, 16);
    cpb = cpb < most ? cpb : most;
    grid = bh * (cpb < PN_MAX_PARTS - 2 ? cpb : PN_MAX_PARTS - 2);
    // one CTA per pair on at most three quarters of the SMs: they cannot draw the bandwidth, and long runs are worth the crossings (80 pairs x
    // 1250 steps: 148.9 us, crossing 134.2; x 563: 73.2 and 66.0; x 188: 27.4 and 30.7; 104 x 563: 84.5 and 82.3, x 188: 34.1 and 34.6; 120 x
    // 563: 93.6 and 94.1)
    if (cpb == 1 && p.spp > 448 && 4 * bh < 3 * sms) grid = sms;
  } else {
    const long long waves = (bh + sms - 1) / sms;
    grid = p.spp > 96 && bh * 5 < waves * sms * 4 ? sms : bh;
  }
  if (grid >= (1ll << 31)) return p;
  p.grid = (int)grid;
  p.slots = G > 8 ? 3 : 4;
  p.off_red = (uint32_t)(PN_WARPS * p.slots) * PN_PIECE;
  p.smem = 1024 + (size_t)p.off_red + sizeof(float) * PN_HALF * (size_t)G * D;
  p.ok = 1;
  return p;
}

PlainWs plain_ws(const kvc_layer* L, int B) {
  PlainWs w{};
  const size_t bh = (size_t)B * L->desc.H_kv, slots = (size_t)part_slots(L, B);
  size_t off = align_up(sizeof(int) * (bh + 1), 256);                  // behind the status word of the layout all paths share
  auto take = [&](size_t bytes) { const size_t o = off; off = align_up(off + bytes, 256); return o; };
  w.off_cnt = take(sizeof(unsigned long long) * bh);
  w.off_pml = take(sizeof(float2) * bh * slots * L->G);
  w.off_py = take(sizeof(float) * bh * slots * L->G * D);
  w.bytes = off;
  return w;
}

template <int NH, int SLOTS>
static cudaError_t launch_plain_inst(const CUtensorMap* tm, const PlainArgs& a, const PlainPlan& p, cudaStream_t st) {
  cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(plain_decode_kernel<NH, SLOTS>), p.smem);
  if (e != cudaSuccess) return e;
  return launch_dependent(plain_decode_kernel<NH, SLOTS>, dim3((unsigned)p.grid), dim3(PN_THREADS), p.smem, st, tm[0], tm[1], tm[2], tm[3], a);
}

cudaError_t launch_plain(const kvc_layer* L, const DecodeArgs& d, const PlainPlan& p, char* ws, cudaStream_t st, bool* encoded) {
  *encoded = false;
  const int B = d.B, H = d.H_kv, S0 = d.R * d.n;
  CUtensorMap tm[4];
  for (int x = 0; x < 2; ++x) {
    // (64 channels, rows, channel half, pairs): a box lands as [half][16 rows][64]; rows past a pair's last are zero-filled
    const int rows = x == 0 ? S0 : d.T, pitch = x == 0 ? S0 : d.T_cap;
    if (rows == 0) continue;
    const uint64_t dims[4] = {64ull, (uint64_t)rows, 2ull, (uint64_t)B * H};
    const uint64_t str[3] = {256ull, 128ull, (uint64_t)pitch * 256};
    const uint32_t box[4] = {64u, (uint32_t)PN_ROWS, 2u, 1u};
    if (!encode_tensor_map_bf16(&tm[2 * x], x == 0 ? d.Kc : d.K_txt, 4, dims, str, box) ||
        !encode_tensor_map_bf16(&tm[2 * x + 1], x == 0 ? d.Vc : d.V_txt, 4, dims, str, box))
      return cudaSuccess;
  }
  if (S0 == 0) { tm[0] = tm[2]; tm[1] = tm[3]; }
  if (d.T == 0) { tm[2] = tm[0]; tm[3] = tm[1]; }
  *encoded = true;
  const PlainWs w = plain_ws(L, B);
  PlainArgs a{};
  a.q = static_cast<const __nv_bfloat16*>(d.q);
  a.out = static_cast<__nv_bfloat16*>(d.out);
  a.py = reinterpret_cast<float*>(ws + w.off_py);
  a.pml = reinterpret_cast<float2*>(ws + w.off_pml);
  a.cnt = reinterpret_cast<unsigned long long*>(ws + w.off_cnt);
  a.token = d.token; a.status = d.status;
  a.G = d.G; a.S0 = S0; a.T = d.T; a.steps_a = p.steps_a; a.spp = p.spp; a.slots = part_slots(L, B); a.total = p.total; a.off_red = p.off_red;
  ProfScope prof(KVC_KERNEL_FUSED, st, KVC_KERNEL_PLAIN);
  return d.G > 8 ? launch_plain_inst<2, 3>(tm, a, p, st) : launch_plain_inst<1, 4>(tm, a, p, st);
}

}  // namespace kvc
