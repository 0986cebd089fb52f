// Cluster decode kernel (see kvc_cluster.cuh) and its host side.
//
// Bound: latency of the hand-overs (scores -> logits -> probabilities -> weights -> values, each a round trip through L2 or shared
// memory per unit); the bytes take a tenth to a third of the time.  Measured on B200: 8 sequences x 5 blocks of n = 729, 28/4 heads,
// 300 text rows: 37.5 us per call (277 us with the three-phase kernels, whose expansion of such block lengths ran on the CUDA cores);
// time line: scores until 5 us, logits 11, probabilities 13, weights 16, joined 20, values 25, merged 27-34.
// Why one kernel of clusters: a unit's CTAs hand S and the partial weights to each other through L2 behind an mbarrier instead of a
// kernel boundary, and while the tensor cores expand, the consumers ask the unit's value rows (and the next unit's key rows) into
// L2, so that HBM does not idle.
// Why warp groups with their own ring slots: a tile is a chain of dependent steps for a warp, so the tiles in work set the pace; a
// group owns its slots (slot mod CL_GROUPS), which keeps a slot's rounds in one group's order.  Why three groups: up to sixteen warps
// have 128 registers a thread; with four groups (eighteen warps, 96 registers) every step spilled, and with the L1 given to shared
// memory a spilled value is an L2 round trip (201 against 151 us at 16 x 8 blocks of n = 1024, both before the steps' registers were
// kept apart).
//
// Roles: warps 0-11 consumers, warp 12 MMA issue, warp 13 TMA producer.
#include <algorithm>
#include <mutex>

#include "kvc_cluster.cuh"
#include "kvc_fused.cuh"
#include "kvc_tcgen05.cuh"

namespace kvc {

constexpr float CL_QSCALE = 0.08838834764831845f * 1.4426950408889634f;      // sigma = 1/sqrt(128), logits in log2 units
constexpr uint32_t CL_QPITCH = 272;                                          // bytes per staged query row (conflict-free ldmatrix)
static_assert((CL_ROWS + 15) * CL_QPITCH <= CL_DUE, "a unit's queries (and the rows a fragment reads past them) in the region of P");
static_assert(CL_ROWS * sizeof(int) <= CL_W_TAIL - CL_DUE && CL_MAX_RAGGED_B < (1 << 16), "the unit's sequences");

struct ClusterBars {
  uint64_t kfull[CL_K_SLOTS], kempty[CL_K_SLOTS];
  uint64_t vfull[CL_V_SLOTS], vempty[CL_V_SLOTS];
  uint64_t xfull[CL_X_SLOTS], xempty[CL_X_SLOTS];
  uint64_t l_done, p_ready, w_done, w_free;
  uint64_t s_ready, w_ready;                                  // cluster-wide: an arrival of every CTA
  uint64_t text[CL_WARPS][CL_TEXT_SLOTS];
};

struct Unit { int h, blk0, nb, nt; };

// A thread's roles, derived anew where a step begins: kept across the loop over units they (and everything the compiler hoists with
// them) took some 100 registers more than a thread has, and with the L1 given to shared memory a spill is an L2 round trip.
struct Lanes { int warp, lane, grp, rg, gid, t4, l7, lmid, lrowB; };
__device__ __forceinline__ Lanes lanes_of(int tid) {
  tid = fresh(tid);
  const int warp = tid >> 5, lane = tid & 31;
  // group, 16-row part of a tile; fragment row and column pair; ldmatrix address pattern: rows 0-7 | 0-7 | 8-15 | 8-15
  return Lanes{warp, lane, warp >> 2, warp & 3, lane >> 2, lane & 3, lane & 7, (lane >> 3) & 1, (lane & 7) + (lane >> 4) * 8};
}

// (sequence, block) of the k-th existing block of a KV head
__device__ __forceinline__ void cl_locate(const ClusterArgs& a, const int* pre, int k, int& b, int& r) {
  if (!pre) { b = k / a.R; r = k - b * a.R; return; }
  int lo = 0, hi = a.B;                                       // pre[lo] <= k < pre[hi]
  while (hi - lo > 1) { const int mid = (lo + hi) >> 1; if (pre[mid] <= k) lo = mid; else hi = mid; }
  b = lo; r = k - pre[lo];
}
// the blocks of a KV head one after the other
struct BlockWalk {
  int b, r, rb;
  __device__ __forceinline__ void start(const ClusterArgs& a, const int* pre, int k) { cl_locate(a, pre, k, b, r); rb = pre ? pre[b + 1] - pre[b] : a.R; }
  __device__ __forceinline__ void next(const ClusterArgs& a, const int* pre) {
    if (++r < rb) return;
    r = 0;
    ++b;
    if (pre) while (b < a.B && (rb = pre[b + 1] - pre[b]) == 0) ++b;
  }
  __device__ __forceinline__ int index(const ClusterArgs& a, int h) const { return (b * a.H_kv + h) * a.R + r; }      // in the capsule store
};
__device__ __forceinline__ int cl_first(const ClusterArgs& a, const int* pre, int b) { return pre ? pre[b] : b * a.R; }
__device__ __forceinline__ int cl_text(const ClusterArgs& a, const int* tx, int b) { return tx ? tx[b] : a.T; }

// The value tiles of a unit are dealt in contiguous runs to its P = CL_GROUPS NS pieces (piece p: CTA p mod NS, group p / NS)
__device__ __forceinline__ int run_start(int p, int nt, int P) { return nt >= P ? p * nt / P : (p < nt ? p : nt); }
__device__ __forceinline__ int run_of(int t, int nt, int P) { return nt >= P ? ((t + 1) * P - 1) / nt : t; }


// Slot x of the value ring's weight slices: the first a.nwp behind the groups' reductions in the region of P, which the slices, asked for
// after w_ready, find free; the others behind the value tiles
__device__ __forceinline__ uint32_t cl_w_slot(const ClusterArgs& a, int x) {
  return x < a.nwp ? CL_W_TAIL + (uint32_t)x * a.w_bytes : CL_P_BYTES + a.w_off + (uint32_t)(x - a.nwp) * a.w_bytes;
}

// What the merge of a (sequence, KV head) has to know about the call's units
struct ClusterView { const int *pre, *tx; UnitSplit us; int nblk; };

// tiles of unit u that belong to a sequence whose blocks are [f0, f1) -> the run of pieces [pa, pa + the result) that hold them
__device__ __forceinline__ int cl_pieces(const ClusterArgs& a, const ClusterView& v, int u, int f0, int f1, int& pa) {
  const int P = CL_GROUPS * a.NS, b0 = u * v.us.rb, nt = min(v.us.rb, v.nblk - b0) * a.vt;
  const int ta = (max(f0, b0) - b0) * a.vt, te = (min(f1, b0 + v.us.rb) - b0) * a.vt;
  pa = run_of(ta, nt, P);
  return run_of(te - 1, nt, P) - pa + 1;
}

// partials a (sequence, KV head) gets in all
__device__ __forceinline__ int cl_expected(const ClusterArgs& a, const ClusterView& v, int b) {
  const int f0 = cl_first(a, v.pre, b), f1 = cl_first(a, v.pre, b + 1);
  int e = (cl_text(a, v.tx, b) + a.tc - 1) / a.tc, pa;
  if (f0 < f1)
    for (int u = f0 / v.us.rb; u <= (f1 - 1) / v.us.rb; ++u) e += cl_pieces(a, v, u, f0, f1, pa);
  return e;
}

// the same by all lanes of a warp, one of the sequence's units each
__device__ __forceinline__ int cl_expected_warp(const ClusterArgs& a, const ClusterView& v, int b) {
  const int f0 = cl_first(a, v.pre, b), f1 = cl_first(a, v.pre, b + 1);
  int e = 0, pa;
  if (f0 < f1)
    for (int u = f0 / v.us.rb + (fresh(threadIdx.x) & 31); u <= (f1 - 1) / v.us.rb; u += 32) e += cl_pieces(a, v, u, f0, f1, pa);
  return __reduce_add_sync(0xffffffffu, e) + (cl_text(a, v.tx, b) + a.tc - 1) / a.tc;
}

// The last partial of a (sequence, KV head) merges: the G query heads of every pair b H_kv + h of list[0 .. n), warps wi of nw taking
// (pair, query head) wi, wi + nw, ...  A lane finds one partial and its statistics; the values are loaded sixteen partials at a time (L2's
// latency bounds it: with 8 in flight and a warp group per sequence the merge of 8 sequences of 5 blocks, 28/4 heads, took 8 us, now 3-6).
__device__ __forceinline__ void cl_merge(const ClusterArgs& a, const ClusterView& v, const int* list, int n, int wi, int nw) {
  const int G = a.G, lane = fresh(threadIdx.x) & 31;
#pragma unroll 1
  for (int e = wi; e < n * G; e += nw) {
    const int i = e / G, g = e - i * G, bh = list[i], b = bh / a.H_kv, h = bh - b * a.H_kv;
    const int f0 = cl_first(a, v.pre, b), f1 = cl_first(a, v.pre, b + 1), u0 = f0 / v.us.rb, u1 = (f1 - 1) / v.us.rb;
    float M = -INFINITY, den = 0.f;
    float4 num = make_float4(0.f, 0.f, 0.f, 0.f);
    int total, p0 = 0;
#pragma unroll 1
    do {
      int k = p0 + lane, slot = -1;
      total = 0;
      if (f0 < f1)
        for (int u = u0; u <= u1; ++u) {
          int pa;
          const int np = cl_pieces(a, v, u, f0, f1, pa);
          if ((unsigned)k < (unsigned)np) slot = h * (v.us.nu * CL_GROUPS * a.NS + a.B) + b + u * CL_GROUPS * a.NS + pa + k;
          k -= np; total += np;
        }
      const int nt = (cl_text(a, v.tx, b) + a.tc - 1) / a.tc;
      if ((unsigned)k < (unsigned)nt) slot = a.tslot0 + (b * a.H_kv + h) * a.nct + k;
      total += nt;
      const float2 st = slot >= 0 ? __ldcg(&a.pml[(size_t)slot * G + g]) : make_float2(-INFINITY, 0.f);
      const int cnt = min(32, total - p0);
      float4 y[16];
      auto load = [&](int p) {
#pragma unroll
        for (int x = 0; x < 16; ++x) {
          const int sl = __shfl_sync(0xffffffffu, slot, p + x);
          y[x] = sl >= 0 ? __ldcg(reinterpret_cast<const float4*>(a.py + ((size_t)sl * G + g) * D + lane * 4)) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
      };
      load(0);
      float mx = st.x;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      mx = fmaxf(mx, M);
      const float f = st.x == -INFINITY ? 0.f : fast_exp2(st.x - mx);
      float d = f * st.y;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
      const float sc = M == -INFINITY ? 0.f : fast_exp2(M - mx);
      M = mx;
      den = fmaf(den, sc, d);
      num.x *= sc; num.y *= sc; num.z *= sc; num.w *= sc;
#pragma unroll 1
      for (int p = 0;;) {
#pragma unroll
        for (int x = 0; x < 16; ++x) {
          const float w = __shfl_sync(0xffffffffu, f, p + x);
          num.x = fmaf(w, y[x].x, num.x); num.y = fmaf(w, y[x].y, num.y); num.z = fmaf(w, y[x].z, num.z); num.w = fmaf(w, y[x].w, num.w);
        }
        if ((p += 16) >= cnt) break;
        load(p);
      }
      p0 += 32;
    } while (p0 < total);
    const float inv = den > 0.f ? 1.f / den : 0.f;
    uint2 o;
    o.x = pack2_bf16(num.x * inv, num.y * inv); o.y = pack2_bf16(num.z * inv, num.w * inv);
    *reinterpret_cast<uint2*>(a.out + ((size_t)bh * G + g) * D + lane * 4) = o;
  }
}

// The list of the pairs a CTA has to merge after its text items, their number in front of it; the list lies in the units' tables, whose
// last use is over by then
__device__ __forceinline__ int* cl_text_due(const ClusterArgs& a, unsigned char* sm) { return reinterpret_cast<int*>(sm + a.tab_off) + 1; }

// Text rows: items of up to tc rows of a (sequence, KV head), a warp each, through the warp's own ring of 16-row pieces (4 KB, keys
// and values in turn), flash-style; the item's partial goes straight from the registers to the workspace.  True if a wait gave up.
template <int NH>
__device__ __forceinline__ bool cl_text_part(const CUtensorMap& tmKt, const CUtensorMap& tmVt, const ClusterArgs& a, const ClusterView& v,
                                             unsigned char* sm, ClusterBars& bars) {
  const Lanes ln = lanes_of(threadIdx.x);
  const int warp = ln.warp, lane = ln.lane, gid = ln.gid, t4 = ln.t4, l7 = ln.l7, lmid = ln.lmid, lrowB = ln.lrowB;
  const int G = a.G, cid = (int)blockIdx.x / a.NS;
  bool dead = false;
  // ---------------- text rows: items of up to tc rows of a (sequence, KV head), a warp each ----------------
  int it, it_end, it_step;
  if (cid < a.ucl) {
    it_step = a.ucl * a.NS * CL_WARPS; it_end = a.text_items;
    it = a.text_ded + warp * a.ucl * a.NS + (int)blockIdx.x;
  } else {
    it_step = (a.ncl - a.ucl) * a.NS * CL_WARPS; it_end = a.text_ded;
    it = warp * (a.ncl - a.ucl) * a.NS + (int)blockIdx.x - a.ucl * a.NS;
  }
  if (it - warp * (it_step / CL_WARPS) >= it_end) return false;      // no item for any warp of the CTA
  unsigned char* tring = sm + (uint32_t)warp * (CL_TEXT_SLOTS * 4096u);
  const uint32_t tring_u = smem_addr(tring);
  auto item_rows = [&](int k, int& b, int& h, int& t0) {
    const int bh = k / a.nct;
    b = bh / a.H_kv; h = bh - b * a.H_kv;
    t0 = (k - bh * a.nct) * a.tc;
    return min(a.tc, cl_text(a, v.tx, b) - t0);
  };
  int is_it = it, is_rg = 0, is_n = -1, is_b = 0, is_h = 0, is_t0 = 0;
  uint32_t is_kv = 0, is_cnt = 0, us_cnt = 0;
  auto issue_next = [&]() {
    if (is_n < 0) {
      while (is_it < it_end && (is_n = item_rows(is_it, is_b, is_h, is_t0)) <= 0) is_it += it_step;
      if (is_it >= it_end) { is_n = -1; return; }
      is_rg = 0; is_kv = 0;
    }
    const uint32_t s = is_cnt % CL_TEXT_SLOTS;
    if (lane == 0) {
      mbar_expect_tx(&bars.text[warp][s], 4096u);
      tma_load_5d(tring + s * 4096u, is_kv ? &tmVt : &tmKt, 0, is_t0 + is_rg * 16, 0, is_h, is_b, &bars.text[warp][s]);
    }
    ++is_cnt;
    is_kv ^= 1u;
    if (is_kv == 0 && ++is_rg * 16 >= is_n) { is_n = -1; is_it += it_step; }
  };
  if (it < it_end && lane == 0) { tma_prefetch_desc(&tmKt); tma_prefetch_desc(&tmVt); }
  for (int x = 0; x < CL_TEXT_SLOTS; ++x) issue_next();
  for (; it < it_end; it += it_step) {
    int b, h, t0;
    const int n_rows = item_rows(it, b, h, t0);
    if (n_rows <= 0) continue;
    const int bh = b * a.H_kv + h;
    uint32_t qa[8][4];
    {
      const __nv_bfloat16* q0 = a.q + (size_t)bh * G * D;
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
    for (int r0 = 0; r0 < n_rows; r0 += 16) {
      const int nv = min(16, n_rows - r0);
      // ---- keys
      uint32_t s = us_cnt % CL_TEXT_SLOTS;
      if (!dead && !mbar_wait_bounded<false>(&bars.text[warp][s], (us_cnt / CL_TEXT_SLOTS) & 1u)) dead = true;
      __syncwarp();
      float cc[2][4];
      {
        float c2[2][2][4];
#pragma unroll
        for (int x = 0; x < 2; ++x)
#pragma unroll
          for (int nt = 0; nt < 2; ++nt)
#pragma unroll
            for (int e = 0; e < 4; ++e) c2[x][nt][e] = 0.f;
        const uint32_t k_u = tring_u + s * 4096u + (uint32_t)lrowB * 128u;
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
          for (int e = 0; e < 4; ++e) cc[nt][e] = c2[0][nt][e] + c2[1][nt][e];
      }
      __syncwarp();
      ++us_cnt;
      issue_next();
#pragma unroll
      for (int nt = 0; nt < 2; ++nt)
#pragma unroll
        for (int e = 0; e < 4; ++e) cc[nt][e] = nt * 8 + 2 * t4 + (e & 1) < nv ? cc[nt][e] * CL_QSCALE : -INFINITY;
      float scl[NH];
#pragma unroll
      for (int hr = 0; hr < NH; ++hr) {
        float mx = fmaxf(fmaxf(cc[0][2 * hr], cc[0][2 * hr + 1]), fmaxf(cc[1][2 * hr], cc[1][2 * hr + 1]));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
        const float m_new = fmaxf(m_run[hr], mx);              // finite: the rows hold at least one valid row
        scl[hr] = fast_exp2(m_run[hr] - m_new);
        m_run[hr] = m_new;
        float ps = 0.f;
#pragma unroll
        for (int nt = 0; nt < 2; ++nt)
#pragma unroll
          for (int x = 0; x < 2; ++x) {
            const float p = fast_exp2(cc[nt][2 * hr + x] - m_new);
            cc[nt][2 * hr + x] = p;
            ps += p;
          }
        l_run[hr] = l_run[hr] * scl[hr] + ps;
      }
#pragma unroll
      for (int nh = 0; nh < NH; ++nh) {
        const float c0s = __shfl_sync(0xffffffffu, scl[nh], (2 * t4) * 4);
        const float c1s = __shfl_sync(0xffffffffu, scl[nh], (2 * t4 + 1) * 4);
        if (c0s != 1.f || c1s != 1.f) {
#pragma unroll
          for (int mt = 0; mt < 8; ++mt) {
            yacc[mt][nh][0] *= c0s; yacc[mt][nh][1] *= c1s;
            yacc[mt][nh][2] *= c0s; yacc[mt][nh][3] *= c1s;
          }
        }
      }
      // ---- values
      s = us_cnt % CL_TEXT_SLOTS;
      if (!dead && !mbar_wait_bounded<false>(&bars.text[warp][s], (us_cnt / CL_TEXT_SLOTS) & 1u)) dead = true;
      __syncwarp();
      const bool ragged_rows = a.T_b != nullptr && nv < 16;
      if (ragged_rows) {
        // rows past the sequence's length may hold anything (rows past T are zero-filled by the copy)
        for (int x = lane; x < (16 - nv) * 16; x += 32) {
          const int rr = nv + (x >> 4), c = x & 15;
          *reinterpret_cast<uint4*>(tring + s * 4096u + (uint32_t)(c >> 3) * 2048u + (uint32_t)rr * 128u + (uint32_t)(c & 7) * 16u) = make_uint4(0, 0, 0, 0);
        }
        __syncwarp();
      }
      {
        uint32_t pb[NH][2], px[NH][2];
#pragma unroll
        for (int nh = 0; nh < NH; ++nh) {
          pb[nh][0] = pack2_bf16(cc[0][2 * nh], cc[0][2 * nh + 1]); pb[nh][1] = pack2_bf16(cc[1][2 * nh], cc[1][2 * nh + 1]);
          px[nh][0] = split_lo(cc[0][2 * nh], cc[0][2 * nh + 1], pb[nh][0]);
          px[nh][1] = split_lo(cc[1][2 * nh], cc[1][2 * nh + 1], pb[nh][1]);
        }
        const uint32_t v_u = tring_u + s * 4096u + (uint32_t)lrowB * 128u;
#pragma unroll
        for (int mt = 0; mt < 8; ++mt) {
          uint32_t av[4];
          ldsm_x4_t(av, v_u + (mt >> 2) * 2048u + (uint32_t)(((((mt & 3) * 2 + lmid)) ^ l7) << 4));
#pragma unroll
          for (int nh = 0; nh < NH; ++nh) {
            mma_bf16_16816(yacc[mt][nh], av, pb[nh][0], pb[nh][1]);
            mma_bf16_16816(yacc[mt][nh], av, px[nh][0], px[nh][1]);
          }
        }
      }
      if (ragged_rows) fence_proxy_async();                    // the zeroed rows before the next copy into this piece
      __syncwarp();
      ++us_cnt;
      issue_next();
    }
    // ---- the item's partial, straight from the registers
    const size_t slot = (size_t)a.tslot0 + (size_t)bh * a.nct + (size_t)(t0 / a.tc);
#pragma unroll
    for (int nh = 0; nh < NH; ++nh) {
      float l = l_run[nh];
      l += __shfl_xor_sync(0xffffffffu, l, 1);
      l += __shfl_xor_sync(0xffffffffu, l, 2);
      if (t4 == 0 && gid + 8 * nh < G) a.pml[slot * G + gid + 8 * nh] = make_float2(m_run[nh], dead ? 0.f : l);
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int head = nh * 8 + 2 * t4 + e;
        if (head < G) {
          float* yp = a.py + (slot * G + head) * D;
#pragma unroll
          for (int mt = 0; mt < 8; ++mt) {
            yp[mt * 16 + gid] = yacc[mt][nh][e];
            yp[mt * 16 + gid + 8] = yacc[mt][nh][2 + e];
          }
        }
      }
    }
    __threadfence();
    __syncwarp();
    const int expected = cl_expected_warp(a, v, b);
    if (lane == 0 && arrive_is_last(&a.cnt[bh], a.token, expected)) {
      __threadfence();
      int* due = cl_text_due(a, sm);
      due[atomicAdd(due - 1, 1)] = bh;
    }
  }
  // The pairs whose last partial was one of the text's, by all warps of the CTA: a warp that merged its own alone took a round trip to L2
  // per query head and sixteen partials, one after the other (2 x 15 blocks of n = 81, 16/1 heads, 338 text rows: 58 us per call,
  // now 31; 28/4 heads, 2 x 15 of n = 81, 1500 rows: 46 and 26)
  named_barrier_sync(1, CL_CONS);
  const int* due = cl_text_due(a, sm);
  cl_merge(a, v, due, due[-1], fresh(threadIdx.x) >> 5, CL_WARPS);
  return dead;
}

template <int NH, int PL>
__global__ void __launch_bounds__(CL_THREADS, 1)
cluster_decode_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
                      const __grid_constant__ CUtensorMap tmKt, const __grid_constant__ CUtensorMap tmVt,
                      const __grid_constant__ CUtensorMap tmS, const __grid_constant__ CUtensorMap tmTh0,
                      const __grid_constant__ CUtensorMap tmTh1, const __grid_constant__ CUtensorMap tmU,
                      const __grid_constant__ CUtensorMap tmWld,
                      const __grid_constant__ ClusterArgs a) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* sm = smem_raw + ((1024u - (smem_addr(smem_raw) & 1023u)) & 1023u);
  __shared__ __align__(8) ClusterBars bars;
  __shared__ uint32_t s_tmem;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  unsigned char* ring = sm + CL_P_BYTES;
  float* rstat = reinterpret_cast<float*>(sm + a.tab_off);                     // [CL_GROUPS][128] maxima, then sums
  float2* tab = reinterpret_cast<float2*>(sm + a.tab_off + CL_GROUPS * 512);   // [NS][128] row (maximum, sum), written by the cluster's CTAs
  const int NS = a.NS, G = a.G;
  const int rank = (int)blockIdx.x % NS, cid = (int)blockIdx.x / NS;
  const bool ragged = a.R_b != nullptr || a.T_b != nullptr;
  int* pre_sm = reinterpret_cast<int*>(sm + a.pre_off);
  const int* pre = a.R_b ? pre_sm : nullptr;                                   // [B + 1] prefix sums of the block counts
  const int* tx = a.T_b ? pre_sm + a.B + 1 : nullptr;                          // [B] text lengths

  if (tid == 0) {
    for (int s = 0; s < CL_K_SLOTS; ++s) { mbar_init(&bars.kfull[s], 1); mbar_init(&bars.kempty[s], 4); }
    for (int s = 0; s < CL_V_SLOTS; ++s) { mbar_init(&bars.vfull[s], 1); mbar_init(&bars.vempty[s], 4); }
    for (int s = 0; s < CL_X_SLOTS; ++s) { mbar_init(&bars.xfull[s], 1); mbar_init(&bars.xempty[s], 1); }
    mbar_init(&bars.l_done, 1); mbar_init(&bars.p_ready, CL_WARPS); mbar_init(&bars.w_done, 1); mbar_init(&bars.w_free, CL_WARPS);
    mbar_init(&bars.s_ready, (uint32_t)NS); mbar_init(&bars.w_ready, (uint32_t)NS);
    for (int w = 0; w < CL_WARPS; ++w)
      for (int s = 0; s < CL_TEXT_SLOTS; ++s) mbar_init(&bars.text[w][s], 1);
    fence_mbar_init();
    cl_text_due(a, sm)[-1] = 0;
  }
  if (warp == CL_WARPS) tmem_alloc(&s_tmem, 512u);
  // per-sequence lengths are inputs like the queries: read after the stream's previous kernel
  if (ragged) {
    grid_dep_wait();
    if (a.T_b && warp == 1)
      for (int b = lane; b < a.B; b += 32) {
        const int t = a.T_b[b];
        pre_sm[a.B + 1 + b] = t < 0 ? 0 : (t > a.T ? a.T : t);
      }
    if (a.R_b && warp == 0) {
      int carry = 0;
      if (lane == 0) pre_sm[0] = 0;
      for (int b0 = 0; b0 < a.B; b0 += 32) {
        const int b = b0 + lane;
        int x = b < a.B ? a.R_b[b] : 0;
        x = x < 0 ? 0 : (x > a.R ? a.R : x);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const int y = __shfl_up_sync(0xffffffffu, x, o); if (lane >= o) x += y; }
        if (b < a.B) pre_sm[b + 1] = carry + x;
        carry += __shfl_sync(0xffffffffu, x, 31);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (NS > 1) cluster_sync_all();                             // the peers' barriers exist before anybody arrives on them
  tc_fence_after();
  const uint32_t tb = s_tmem;

  const int nblk = pre ? pre[a.B] : a.B * a.R;                // existing blocks of a KV head
  const UnitSplit us = split_units(nblk, a.rbmax, a.cap);
  const int units = cid < a.ucl ? a.H_kv * us.nu : 0;
  auto unit_at = [&](int w) {
    Unit u;
    u.h = w / us.nu;
    u.blk0 = (w - u.h * us.nu) * us.rb;
    u.nb = min(us.rb, nblk - u.blk0);
    u.nt = u.nb * a.vt;
    return u;
  };
  const int P = CL_GROUPS * NS;
  // this CTA's columns: groups [g0, g1) of 64
  const int cg0 = rank * a.ncg / NS, ngrp = (rank + 1) * a.ncg / NS - cg0;
  const int NWc = ngrp * 64;

  if (warp == CL_WARPS + 1) {
    // =========================================== producer ===========================================
    if (lane == 0 && units > 0) {
      tma_prefetch_desc(&tmK); tma_prefetch_desc(&tmTh0); tma_prefetch_desc(&tmTh1); tma_prefetch_desc(&tmU);
      tma_prefetch_desc(&tmS); tma_prefetch_desc(&tmV); tma_prefetch_desc(&tmWld);
      const CUtensorMap* tmTh = ngrp * NS >= a.ncg ? &tmTh0 : &tmTh1;          // boxes of ceil(ncg / NS) groups, or one less
      // Every phase of a unit starts at slot 0 of its ring.  Bit s of a ring's word: the parity of the number of fills of slot s; the
      // last one has been consumed when the slot's empty barrier has left that parity's phase (a slot never filled passes at once).
      uint32_t kb = 0, vb = 0, xb = 0;
      bool ok = true;
      auto drained = [&](uint64_t* empty, uint32_t bits, int s) { if (ok && !mbar_wait_bounded(&empty[s], ((bits >> s) & 1u) ^ 1u)) ok = false; };
      bool waited = ragged;
      if (!a.early && !waited) { grid_dep_wait(); waited = true; }
      const int spg = a.nV / CL_GROUPS;                                       // value slots per group
      const int kc0 = cid % a.nk1;      // chunks are walked from a different start by every cluster: not all ask L2 for the same lines at once
      const uint32_t th_bytes = (uint32_t)NWc * 128u;
      uint32_t round = 0;
      for (int w = cid; w < units && ok; w += a.ucl, ++round) {
        const Unit u = unit_at(w);
        // ---- step 1: this CTA's key tiles; tile i to slot i mod nK (a multiple of CL_GROUPS), whose memory the last unit's value tiles held
        {
          int bl = rank / a.vt, jt = rank - bl * a.vt, x = 0, vd = 0;
          BlockWalk bw;
          bw.start(a, pre, u.blk0 + bl);
          for (int t = rank; t < u.nt && ok; t += NS) {
            drained(bars.kempty, kb, x);
            if (round > 0) while (vd < a.nV && (vd <= x || x >= a.nV)) drained(bars.vempty, vb, vd++);
            if (!ok) break;
            kb ^= 1u << x;
            mbar_expect_tx(&bars.kfull[x], CL_TILE_BYTES);
            tma_load_4d(ring + x * CL_TILE_BYTES, &tmK, 0, jt * CL_TILE, 0, bw.index(a, u.h), &bars.kfull[x]);
            if (++x == a.nK) x = 0;
            jt += NS;
            while (jt >= a.vt) { jt -= a.vt; bw.next(a, pre); }
          }
          if (round > 0) while (vd < a.nV) drained(bars.vempty, vb, vd++);
        }
        if (!waited) { grid_dep_wait(); waited = true; }
        // ---- step 2: theta chunks; the scores of the unit's other CTAs are complete once s_ready turns (and then this CTA's consumers
        // have left its key tiles)
        const int npre = a.nk1 < a.nX ? a.nk1 : a.nX;
        int kc = kc0, kd = 0;
        for (int i = 0; i < npre && ok; ++i) {
          const uint32_t end = (uint32_t)(i + 1) * a.x_bytes;
          drained(bars.xempty, xb, i);
          while (kd < a.nK && (uint32_t)kd * CL_TILE_BYTES < end) drained(bars.kempty, kb, kd++);
          if (!ok) break;
          xb ^= 1u << i;
          mbar_expect_tx(&bars.xfull[i], a.s_bytes + th_bytes);
          tma_load_4d(ring + (uint32_t)i * a.x_bytes + a.s_bytes, tmTh, 0, kc * 64, cg0, u.h, &bars.xfull[i]);
          kc = kc + 1 < a.nk1 ? kc + 1 : 0;
        }
        if (ok && !mbar_wait_cluster_bounded(&bars.s_ready, round & 1u)) ok = false;
        fence_proxy_async_all();
        if (!ok) break;
        for (int i = 0, k = kc0; i < npre; ++i) {
          tma_load_4d(ring + (uint32_t)i * a.x_bytes, &tmS, k * 64, 0, 0, cid, &bars.xfull[i]);
          k = k + 1 < a.nk1 ? k + 1 : 0;
        }
        int xs = npre == a.nX ? 0 : npre;
        for (int i = npre; i < a.nk1 && ok; ++i) {
          drained(bars.xempty, xb, xs);
          if (!ok) break;
          xb ^= 1u << xs;
          unsigned char* dst = ring + (uint32_t)xs * a.x_bytes;
          mbar_expect_tx(&bars.xfull[xs], a.s_bytes + th_bytes);
          tma_load_4d(dst, &tmS, kc * 64, 0, 0, cid, &bars.xfull[xs]);
          tma_load_4d(dst + a.s_bytes, tmTh, 0, kc * 64, cg0, u.h, &bars.xfull[xs]);
          kc = kc + 1 < a.nk1 ? kc + 1 : 0;
          if (++xs == a.nX) xs = 0;
        }
        // ---- step 3: U chunks
        for (int wp = 0; wp < a.npass && ok; ++wp)
          for (int k = 0; k < ngrp && ok; ++k)
            for (int bx = 0; bx < a.nbox && ok; ++bx) {
              drained(bars.xempty, xb, xs);
              if (!ok) break;
              xb ^= 1u << xs;
              mbar_expect_tx(&bars.xfull[xs], (uint32_t)a.brow * 128u);
              tma_load_3d(ring + (uint32_t)xs * a.x_bytes, &tmU, (cg0 + k) * 64, wp * a.prow + bx * a.brow, u.h, &bars.xfull[xs]);
              if (++xs == a.nX) xs = 0;
            }
        // ---- step 4: value tiles with their slices of the partial weights; tile i of group g to slot g + CL_GROUPS (i mod spg).  The
        // first tile of every slot is asked for before the weights are complete (w_ready), as the expansion's slots drain
        int vt0[CL_GROUPS], vn[CL_GROUPS], vj[CL_GROUPS], vbl[CL_GROUPS], most = 0;
        BlockWalk bw[CL_GROUPS];
#pragma unroll
        for (int g = 0; g < CL_GROUPS; ++g) {
          vt0[g] = run_start(g * NS + rank, u.nt, P);
          vn[g] = run_start(g * NS + rank + 1, u.nt, P) - vt0[g];
          most = max(most, vn[g]);
          vbl[g] = vt0[g] / a.vt;
          vj[g] = vt0[g] - vbl[g] * a.vt;
          if (vn[g] > 0) bw[g].start(a, pre, u.blk0 + vbl[g]);
        }
        auto w_slice = [&](int x, int jt, int bl) {
          tma_load_4d(sm + cl_w_slot(a, x), &tmWld, jt * CL_TILE, bl * G, 0, cid, &bars.vfull[x]);
        };
        const int first = most < spg ? most : spg;
        int xd = 0, xg = 0;                                                   // xg: slot of a group's next tile
        for (int i = 0; i < most && ok; ++i) {
#pragma unroll
          for (int g = 0; g < CL_GROUPS; ++g) {
            if (i < vn[g] && ok) {
              const int x = g + CL_GROUPS * xg;
              drained(bars.vempty, vb, x);
              if (i < first) while (xd < a.nX && (uint32_t)xd * a.x_bytes < (uint32_t)(x + 1) * CL_TILE_BYTES) drained(bars.xempty, xb, xd++);
              if (ok) {
                vb ^= 1u << x;
                mbar_expect_tx(&bars.vfull[x], CL_TILE_BYTES + a.w_tx);
                tma_load_4d(ring + x * CL_TILE_BYTES, &tmV, 0, vj[g] * CL_TILE, 0, bw[g].index(a, u.h), &bars.vfull[x]);
                if (i >= first) w_slice(x, vj[g], vbl[g]);
                if (++vj[g] == a.vt) { vj[g] = 0; ++vbl[g]; if (i + 1 < vn[g]) bw[g].next(a, pre); }
              }
            }
          }
          if (++xg == spg) xg = 0;
          if (i == first - 1 && ok) {
            if (!mbar_wait_cluster_bounded(&bars.w_ready, round & 1u)) { ok = false; break; }
            fence_proxy_async_all();
#pragma unroll
            for (int g = 0; g < CL_GROUPS; ++g) {
              int bl = vt0[g] / a.vt, jt = vt0[g] - bl * a.vt;
              for (int x = 0; x < first && x < vn[g]; ++x) {
                w_slice(g + CL_GROUPS * x, jt, bl);
                if (++jt == a.vt) { jt = 0; ++bl; }
              }
            }
          }
        }
        if (most == 0 && ok && !mbar_wait_cluster_bounded(&bars.w_ready, round & 1u)) ok = false;
      }
      if (!waited) grid_dep_wait();
      if (!ok) atomicExch(a.status, (int)KVC_ERR_TIMEOUT);
    }
  } else if (warp == CL_WARPS) {
    // =========================================== MMA issue ===========================================
    const int kc0 = cid % a.nk1;
    const uint32_t ring_u = smem_addr(ring), p_u = smem_addr(sm);
    const uint32_t idesc_L = umma_idesc_bf16(128, NWc, 0, 1);
    const uint32_t idesc_W = umma_idesc_bf16(128, a.brow, 0, 0);
    const uint64_t a0 = umma_smem_desc(ring_u, 16u, 1024u, UMMA_LAYOUT_SW128);                      // S chunk (K-major) / U chunk as B
    const uint64_t b0 = umma_smem_desc(ring_u + a.s_bytes, 8192u, 1024u, UMMA_LAYOUT_SW128);       // theta chunk (MN-major)
    const uint64_t p0 = umma_smem_desc(p_u, 16u, 1024u, UMMA_LAYOUT_SW128);                        // probabilities (K-major)
    const uint64_t lo_S = (uint64_t)((uint32_t)a.srows * 128u >> 4);                               // second term of S
    const uint64_t lo_P = (uint64_t)(((uint32_t)NWc * 256u) >> 4);                                 // second term of P
    uint32_t xs = 0, xb = 0, round = 0, wpass = 0;              // bit s of xb: parity of the fills of slot s taken so far
    bool dead = false;
    auto wait_on = [&](uint64_t* bar, uint32_t parity) {
      if (!dead && !mbar_wait_bounded(bar, parity)) dead = true;
      __syncwarp();
      tc_fence_after();
    };
    for (int w = cid; w < units; w += a.ucl, ++round) {
      int k = kc0;
      xs = 0;
      for (int i = 0; i < a.nk1; ++i) {
        wait_on(&bars.xfull[xs], (xb >> xs) & 1u);
        xb ^= 1u << xs;
        if (lane == 0 && !dead) {
          const uint64_t off = (uint64_t)((xs * a.x_bytes) >> 4);
          const int ksteps = min(4, (a.m - k * 64 + 15) >> 4);
          for (int ks = 0; ks < ksteps; ++ks) {
            umma_bf16(tb, a0 + off + (uint64_t)(ks * 2), b0 + off + (uint64_t)(ks * 128), idesc_L, (i | ks) ? 1u : 0u);
            if (PL == 2) umma_bf16(tb, a0 + off + lo_S + (uint64_t)(ks * 2), b0 + off + (uint64_t)(ks * 128), idesc_L, 1u);
          }
          umma_commit(&bars.xempty[xs]);
          if (i == a.nk1 - 1) umma_commit(&bars.l_done);
        }
        __syncwarp();
        if (++xs == (uint32_t)a.nX) xs = 0;
        k = k + 1 < a.nk1 ? k + 1 : 0;
      }
      wait_on(&bars.p_ready, round & 1u);
      for (int wp = 0; wp < a.npass; ++wp) {
        if (wp > 0) { wait_on(&bars.w_free, wpass & 1u); ++wpass; }
        for (int g = 0; g < ngrp; ++g)
          for (int bx = 0; bx < a.nbox; ++bx) {
            wait_on(&bars.xfull[xs], (xb >> xs) & 1u);
            xb ^= 1u << xs;
            if (lane == 0 && !dead) {
              const uint64_t off = (uint64_t)((xs * a.x_bytes) >> 4), pg = p0 + (uint64_t)(g * (16384 >> 4));
#pragma unroll
              for (int ks = 0; ks < 4; ++ks) {
                umma_bf16(tb + (uint32_t)(bx * a.brow), pg + (uint64_t)(ks * 2), a0 + off + (uint64_t)(ks * 2), idesc_W, (g | ks) ? 1u : 0u);
                if (PL == 2) umma_bf16(tb + (uint32_t)(bx * a.brow), pg + lo_P + (uint64_t)(ks * 2), a0 + off + (uint64_t)(ks * 2), idesc_W, 1u);
              }
              umma_commit(&bars.xempty[xs]);
              if (g == ngrp - 1 && bx == a.nbox - 1) umma_commit(&bars.w_done);
            }
            __syncwarp();
            if (++xs == (uint32_t)a.nX) xs = 0;
          }
      }
    }
    if (dead && lane == 0) atomicExch(a.status, (int)KVC_ERR_TIMEOUT);
  } else {
    // =========================================== consumers ===========================================
    // the parameters of the first unit into L2 (fixed at inference, so before the wait), a share by each of the head's clusters.  Lengths
    // on the device may give fewer units than the clusters launched for them: those without one have no head either
    if (cid < units) {
      const int h = cid / us.nu, lines = a.m * ngrp, step = min(us.nu, a.ucl) * CL_CONS;
      for (int x = (cid - h * us.nu) * CL_CONS + tid; x < lines; x += step) {
        const int row = x / ngrp, c = cg0 + x - row * ngrp;
        prefetch_l2(a.theta + ((size_t)h * a.m + row) * a.theta_np + (size_t)c * 64);
        prefetch_l2(a.U + ((size_t)h * a.m + row) * a.U_np + (size_t)c * 64);
      }
    }
    if (!ragged) grid_dep_wait();
    grid_dep_launch();
    if (blockIdx.x == 0) {
      if (tid == 0) *a.status = 0;
      if (ragged) {
        named_barrier_sync(1, CL_CONS);
        for (int b = tid; b < a.B; b += CL_CONS) {
          const bool bad = (a.R_b && (a.R_b[b] < 0 || a.R_b[b] > a.R)) || (a.T_b && (a.T_b[b] < 0 || a.T_b[b] > a.T));
          if (bad) atomicExch(a.status, (int)KVC_ERR_BOUNDS);
        }
        // sequences without any row: a zero output row
        for (int b = 0; b < a.B; ++b)
          if (cl_first(a, pre, b + 1) == cl_first(a, pre, b) && cl_text(a, tx, b) == 0)
            for (int x = tid; x < a.H_kv * G * (D / 8); x += CL_CONS)
              reinterpret_cast<uint4*>(a.out + (size_t)b * a.H_kv * G * D)[x] = make_uint4(0, 0, 0, 0);
      }
    }
    bool dead = false;

    const ClusterView view{pre, tx, us, nblk};
    uint32_t round = 0, wpass = 0;
    // Hand-over to the cluster's CTAs: everything the consumers have written so far, by one arrival per CTA.  The CTA's barrier and one
    // thread's fence order it (a fence and NS arrivals by every warp took 4 us instead of 2); the readers' proxy fence follows their wait.
    auto tell_cluster = [&](uint64_t* bar) {
      named_barrier_sync(1, CL_CONS);
      if (fresh(tid) < NS) {
        asm volatile("fence.acq_rel.cluster;\n" ::: "memory");
        mbar_arrive_remote(map_to_cta(smem_addr(bar), (uint32_t)fresh(tid)));
      }
    };
    uint32_t kb = 0, vb = 0;                                    // bit s: parity of the fills of slot s taken so far
    // line gt of a 64-row tile of a capsule store into L2 (gt: thread of the group)
    auto prefetch_tile = [&](const __nv_bfloat16* store, int blk, int jt, int gt) {
      if (jt * CL_TILE + (gt >> 1) < a.m) prefetch_l2(store + ((size_t)blk * a.m + jt * CL_TILE) * D + gt * 64);
    };
    for (int w = cid; w < units; w += a.ucl, ++round) {
      const Unit u = unit_at(w);
      const int rows = u.nb * G;
      // ---------------- queries of the unit's sequences ----------------
      // A sequence's G rows lie where its first block's expansion rows are: within the unit's 128 rows whatever lies between its sequences
      // (with per-sequence lengths there may be any number without a block)
      int* ndue = reinterpret_cast<int*>(sm + a.tab_off + CL_GROUPS * 512 + (uint32_t)NS * CL_ROWS * 8u + CL_GROUPS * 64);
      int* nseq_sm = ndue + 1;
      int* seq_sm = reinterpret_cast<int*>(sm + CL_DUE);        // (sequence, its first block of the unit) in any order
      if (fresh(tid) == 0) *nseq_sm = 0;
      named_barrier_sync(1, CL_CONS);                           // the region of P is free (last unit's reductions)
      if (fresh(tid) == 0) *ndue = 0;
      int b_first, nseq, rr_;
      if (pre) {
        if (fresh(tid) < u.nb) {
          int b, r;
          cl_locate(a, pre, u.blk0 + fresh(tid), b, r);
          if (r == 0 || fresh(tid) == 0) seq_sm[atomicAdd(nseq_sm, 1)] = b | fresh(tid) << 16;
        }
        named_barrier_sync(1, CL_CONS);
        b_first = 0;
        nseq = *nseq_sm;
      } else {
        cl_locate(a, pre, u.blk0, b_first, rr_);
        nseq = (u.blk0 + u.nb - 1) / a.R - b_first + 1;
      }
      for (int x = tid; x < nseq * G * 16; x += CL_CONS) {
        const int row = x >> 4, c = x & 15, k = row / G, g = row - k * G;
        const int b = pre ? seq_sm[k] & 0xffff : b_first + k, blk = pre ? seq_sm[k] >> 16 : max(b * a.R - u.blk0, 0);
        *reinterpret_cast<uint4*>(sm + (uint32_t)(blk * G + g) * CL_QPITCH + c * 16) =
            __ldg(reinterpret_cast<const uint4*>(a.q + (((size_t)b * a.H_kv + u.h) * G + g) * D + c * 8));
      }
      named_barrier_sync(1, CL_CONS);
      // ---------------- step 1: scores ----------------
      {
        const auto [warp, lane, grp, rg, gid, t4, l7, lmid, lrowB] = lanes_of(tid);
        const uint32_t sm_u = (uint32_t)fresh((int)smem_addr(sm)), ring_u = sm_u + CL_P_BYTES;
        uint32_t qa[8][4];
        int cur_b = -1;
        __nv_bfloat16* S0 = a.S + (size_t)cid * PL * a.srows * a.ms;
        const int t0 = rank + grp * NS;
        int bl = t0 / a.vt, jt = t0 - bl * a.vt;
        BlockWalk bw;
        if (t0 < u.nt) bw.start(a, pre, u.blk0 + bl);
        int s = grp;
        for (int t = t0; t < u.nt; t += P) {
          const int b = bw.b;
          if (b != cur_b) {
            cur_b = b;
            const uint32_t qrow = sm_u + (uint32_t)((bl - min(bw.r, bl)) * G + (lane & 15)) * CL_QPITCH + (uint32_t)(lane >> 4) * 16u;
#pragma unroll
            for (int ks = 0; ks < 8; ++ks) ldsm_x4(qa[ks], qrow + (uint32_t)ks * 32u);
          }
          if (!dead && !mbar_wait_bounded(&bars.kfull[s], (kb >> s) & 1u)) dead = true;
          kb ^= 1u << s;
          __syncwarp();
          const uint32_t k_u = ring_u + s * CL_TILE_BYTES;
          const int j0 = jt * CL_TILE + rg * 16;
          if (j0 < a.m) {
            float cc[2][2][4];
#pragma unroll
            for (int x = 0; x < 2; ++x)
#pragma unroll
              for (int nt = 0; nt < 2; ++nt)
#pragma unroll
                for (int e = 0; e < 4; ++e) cc[x][nt][e] = 0.f;
            const uint32_t rowB = (uint32_t)((rg * 16 + lrowB) * 128);
#pragma unroll
            for (int ks = 0; ks < 8; ++ks) {
              uint32_t bk[4];
              ldsm_x4(bk, k_u + (ks >> 2) * CL_HALF + rowB + (uint32_t)(((((ks & 3) * 2 + lmid)) ^ l7) << 4));
              mma_bf16_16816(cc[ks & 1][0], qa[ks], bk[0], bk[1]);
              mma_bf16_16816(cc[ks & 1][1], qa[ks], bk[2], bk[3]);
            }
            // cc[.][nt][e]: head gid + 8 (e >> 1), key row j0 + 8 nt + 2 t4 + (e & 1)
#pragma unroll
            for (int hh = 0; hh < NH; ++hh) {
              const int head = gid + 8 * hh;
              if (head < G) {
                __nv_bfloat16* row = S0 + (size_t)(bl * G + head) * a.ms;
#pragma unroll
                for (int nt = 0; nt < 2; ++nt) {
                  const int j = j0 + nt * 8 + 2 * t4;
                  if (j < a.m) {
                    const float v0 = (cc[0][nt][2 * hh] + cc[1][nt][2 * hh]) * CL_QSCALE;
                    const float v1 = (cc[0][nt][2 * hh + 1] + cc[1][nt][2 * hh + 1]) * CL_QSCALE;
                    const uint32_t hi = pack2_bf16(v0, v1);
                    *reinterpret_cast<uint32_t*>(row + j) = hi;
                    if (PL == 2) *reinterpret_cast<uint32_t*>(row + (size_t)a.srows * a.ms + j) = split_lo(v0, v1, hi);
                  }
                }
              }
            }
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(&bars.kempty[s]);
          s = s + CL_GROUPS < a.nK ? s + CL_GROUPS : grp;
          jt += P;
          while (jt >= a.vt) { jt -= a.vt; ++bl; if (bl < u.nb) bw.next(a, pre); }
        }
        tell_cluster(&bars.s_ready);
      }
      // the value tiles this group will take into L2 while the expansions run (HBM has nothing else to do)
      {
        const auto [warp, lane, grp, rg, gid, t4, l7, lmid, lrowB] = lanes_of(tid);
        const int piece = grp * NS + rank;
        const int v0 = run_start(piece, u.nt, P), v1 = run_start(piece + 1, u.nt, P);
        int bl = v0 / a.vt, jt = v0 - bl * a.vt;
        BlockWalk bw;
        if (v0 < v1) bw.start(a, pre, u.blk0 + bl);
        for (int t = v0; t < v1; ++t) {
          prefetch_tile(a.Vc, bw.index(a, u.h), jt, rg * 32 + lane);
          if (++jt == a.vt) { jt = 0; if (t + 1 < v1) bw.next(a, pre); }
        }
      }
      // ---------------- softmax over this CTA's columns: lane <-> row, a third of the columns per warp ----------------
      {
        const auto [warp, lane, grp, rg, gid, t4, l7, lmid, lrowB] = lanes_of(tid);
        const int row = rg * 32 + lane, hf = grp;
        const uint32_t trow = tb + ((uint32_t)(rg * 32) << 16);
        const bool work = rg * 32 < rows;
        unsigned char* sm_p = sm;
        if (!dead && !mbar_wait_bounded(&bars.l_done, round & 1u)) dead = true;
        __syncwarp();
        tc_fence_after();
        const int cb = (hf * (NWc >> 5) / CL_GROUPS) * 32, ce = ((hf + 1) * (NWc >> 5) / CL_GROUPS) * 32;
        const int valid = a.n - cg0 * 64;                       // columns of the range that exist
        float mx = -INFINITY;
        // 32 columns per load, used at once: with the next load in flight as well, the registers of both spilled
        auto columns = [&](auto use) {
#pragma unroll 1
          for (int c0 = cb; c0 < ce; c0 += 32) {
            uint32_t v[32];
            tmem_ld_issue_x32(trow + (uint32_t)c0, v);
            tmem_ld_wait_x32(v);
            use(c0, v);
          }
        };
        if (work) {
          columns([&](int c0, const uint32_t (&v)[32]) {
            if (c0 + 32 <= valid) {
#pragma unroll
              for (int k = 0; k < 32; ++k) mx = fmaxf(mx, __uint_as_float(v[k]));
            } else {
#pragma unroll
              for (int k = 0; k < 32; ++k) mx = fmaxf(mx, c0 + k < valid ? __uint_as_float(v[k]) : -INFINITY);
            }
          });
          rstat[hf * 128 + row] = mx;
        }
        named_barrier_sync(1, CL_CONS);
        if (work) {
#pragma unroll
          for (int x = 0; x < CL_GROUPS; ++x) mx = fmaxf(mx, rstat[x * 128 + row]);
        }
        named_barrier_sync(1, CL_CONS);
        float sum = 0.f;
        if (work) {
          columns([&](int c0, const uint32_t (&v)[32]) {
            unsigned char* g = sm_p + (uint32_t)(c0 >> 6) * 16384u + (uint32_t)row * 128u;
            const int pc = (c0 & 63) >> 3;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              uint32_t hi[4], lo[4];
#pragma unroll
              for (int k = 0; k < 4; ++k) {
                const int c = 8 * q + 2 * k;
                float e0 = fast_exp2(__uint_as_float(v[c]) - mx), e1 = fast_exp2(__uint_as_float(v[c + 1]) - mx);
                if (c0 + c >= valid) e0 = 0.f;
                if (c0 + c + 1 >= valid) e1 = 0.f;
                sum += e0 + e1;
                hi[k] = pack2_bf16(e0, e1);
                if (PL == 2) lo[k] = split_lo(e0, e1, hi[k]);
              }
              const uint32_t at = (uint32_t)(((pc + q) ^ (row & 7)) << 4);
              *reinterpret_cast<uint4*>(g + at) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
              if (PL == 2) *reinterpret_cast<uint4*>(g + (uint32_t)NWc * 256u + at) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
            }
          });
          rstat[hf * 128 + row] = sum;
        }
        fence_proxy_async();                                    // P is read by the tensor core
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars.p_ready);
        named_barrier_sync(1, CL_CONS);
        if (hf == 0 && row < rows) {
          sum = 0.f;
#pragma unroll
          for (int x = 0; x < CL_GROUPS; ++x) sum += rstat[x * 128 + row];
          const uint32_t at = smem_addr(&tab[rank * CL_ROWS + row]);
          for (int c = 0; c < NS; ++c) st_cluster_f32x2(map_to_cta(at, (uint32_t)c), mx, sum);      // (visible with w_ready)
        }
      }
      // the next unit's key tiles into L2 while the second product runs
      if (w + a.ucl < units) {
        const auto [warp, lane, grp, rg, gid, t4, l7, lmid, lrowB] = lanes_of(tid);
        const Unit nx = unit_at(w + a.ucl);
        const int t0 = rank + grp * NS;
        int bl = t0 / a.vt, jt = t0 - bl * a.vt;
        BlockWalk bw;
        if (t0 < nx.nt) bw.start(a, pre, nx.blk0 + bl);
        for (int t = t0; t < nx.nt; t += P) {
          prefetch_tile(a.Kc, bw.index(a, nx.h), jt, rg * 32 + lane);
          jt += P;
          while (jt >= a.vt) { jt -= a.vt; ++bl; if (bl < nx.nb) bw.next(a, pre); }
        }
      }
      // ---------------- the partial weights of the range to the workspace ----------------
      for (int wp = 0; wp < a.npass; ++wp) {
        const auto [warp, lane, grp, rg, gid, t4, l7, lmid, lrowB] = lanes_of(tid);
        const int row = rg * 32 + lane, hf = grp;
        const uint32_t trow = tb + ((uint32_t)(rg * 32) << 16);
        const bool work = rg * 32 < rows;
        if (!dead && !mbar_wait_bounded(&bars.w_done, wpass & 1u)) dead = true;
        ++wpass;
        __syncwarp();
        tc_fence_after();
        const int j0 = wp * a.prow;
        if (work) {
          // A step is 128 bytes of every row, alternating over the column warps.  In the last pass the region of P is free: the rows
          // are turned through it so that a store instruction covers four rows of 128 bytes (a lane storing its own row in 16-byte
          // pieces writes half sectors: 5 us instead of 2 at 128 x 410)
          constexpr int EB = 4, CWD = 128 / EB;
          const bool last = wp == a.npass - 1;
          unsigned char* stage = sm + (uint32_t)warp * 4096u;
          unsigned char* wrow = reinterpret_cast<unsigned char*>(a.W) + (((size_t)cid * NS + rank) * a.srows + rg * 32) * a.ms * EB;
          const int jend = min(a.ms, j0 + a.prow);
          for (int c0 = hf * CWD; j0 + c0 < jend; c0 += CL_GROUPS * CWD) {
#pragma unroll
            for (int cc = 0; cc < CWD; cc += 32) {
              uint32_t v[32];
              tmem_ld_issue_x32(trow + (uint32_t)(c0 + cc), v);
              tmem_ld_wait_x32(v);
#pragma unroll
              for (int q = 0; q < 32 * EB / 16; ++q) {
                const uint4 x = make_uint4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
                const int piece = cc * EB / 16 + q, j = j0 + c0 + piece * (16 / EB);
                if (last) *reinterpret_cast<uint4*>(stage + swz(lane, piece)) = x;
                else if (row < rows && j < jend) *reinterpret_cast<uint4*>(wrow + ((size_t)lane * a.ms + j) * EB) = x;
              }
            }
            if (last) {
              __syncwarp();
              const int j = j0 + c0 + (lane & 7) * (16 / EB);
#pragma unroll
              for (int q = 0; q < 8; ++q) {
                const int rr = q * 4 + (lane >> 3);
                const uint4 x = *reinterpret_cast<const uint4*>(stage + swz(rr, lane & 7));
                if (rg * 32 + rr < rows && j < jend) *reinterpret_cast<uint4*>(wrow + ((size_t)rr * a.ms + j) * EB) = x;
              }
              __syncwarp();
            }
          }
        }
        tc_fence_before();
        __syncwarp();
        if (wp + 1 < a.npass && lane == 0) mbar_arrive(&bars.w_free);
      }
      tell_cluster(&bars.w_ready);
      // ---------------- step 4: the group's run of value tiles ----------------
      if (!dead && !mbar_wait_cluster_bounded(&bars.w_ready, round & 1u)) dead = true;
      __syncwarp();
      {
        const auto [warp, lane, grp, rg, gid, t4, l7, lmid, lrowB] = lanes_of(tid);
        const uint32_t ring_u = (uint32_t)fresh((int)smem_addr(sm)) + CL_P_BYTES;
        const int piece = grp * NS + rank, gt = rg * 32 + lane;
        const int v0 = run_start(piece, u.nt, P), v1 = run_start(piece + 1, u.nt, P);
        float yacc[8][NH][4];
        float m_run[NH], l_run[NH], f[NH][CL_MAX_NS];
        auto reset = [&]() {
#pragma unroll
          for (int nh = 0; nh < NH; ++nh) {
            m_run[nh] = -INFINITY; l_run[nh] = 0.f;
#pragma unroll
            for (int x = 0; x < CL_MAX_NS; ++x) f[nh][x] = 0.f;
#pragma unroll
            for (int mt = 0; mt < 8; ++mt)
#pragma unroll
              for (int e = 0; e < 4; ++e) yacc[mt][nh][e] = 0.f;
          }
        };
        reset();
        int bl = v0 / a.vt, jt = v0 - bl * a.vt;
        int cur_b = -1, s = grp, nflush = 0;
        int mine = 0;                                           // thread x of the group arrives for the run's x-th sequence
        int* due = reinterpret_cast<int*>(sm + CL_DUE);         // pairs this CTA has to merge
        BlockWalk bw;
        if (v0 < v1) bw.start(a, pre, u.blk0 + bl);
        for (int t = v0; t < v1; ++t) {
          if (t == v0 || jt == 0) {
            cur_b = bw.b;
            // a new block: the reference maximum of its rows, the running state rescaled to it, the ranges' factors
            float scl[NH];
#pragma unroll
            for (int nh = 0; nh < NH; ++nh) {
              const int g = gid + 8 * nh;
              scl[nh] = 1.f;
              if (g < G) {
                const float2* tr = tab + bl * G + g;
                float mb = m_run[nh];
#pragma unroll
                for (int s = 0; s < CL_MAX_NS; ++s) if (s < NS) mb = fmaxf(mb, tr[s * CL_ROWS].x);
                scl[nh] = fast_exp2(m_run[nh] - mb);
                m_run[nh] = mb;
                float mass = 0.f;
#pragma unroll
                for (int s = 0; s < CL_MAX_NS; ++s) {
                  f[nh][s] = 0.f;
                  if (s < NS) {
                    const float2 st = tr[s * CL_ROWS];
                    f[nh][s] = fast_exp2(st.x - mb);
                    mass = fmaf(f[nh][s], st.y, mass);
                  }
                }
                // the block's probability mass (and with it the mu term) is counted with its first tile
                l_run[nh] = fmaf(l_run[nh], scl[nh], jt == 0 ? mass : 0.f);
              }
            }
#pragma unroll
            for (int nh = 0; nh < NH; ++nh) {
              const float c0s = __shfl_sync(0xffffffffu, scl[nh], (2 * t4) * 4);
              const float c1s = __shfl_sync(0xffffffffu, scl[nh], (2 * t4 + 1) * 4);
              if (c0s != 1.f || c1s != 1.f) {
#pragma unroll
                for (int mt = 0; mt < 8; ++mt) {
                  yacc[mt][nh][0] *= c0s; yacc[mt][nh][1] *= c1s;
                  yacc[mt][nh][2] *= c0s; yacc[mt][nh][3] *= c1s;
                }
              }
            }
          }
          if (!dead && !mbar_wait_bounded(&bars.vfull[s], (vb >> s) & 1u)) dead = true;
          vb ^= 1u << s;
          __syncwarp();
          if (jt * CL_TILE + rg * 16 < a.m) {
            const unsigned char* wp = sm + cl_w_slot(a, s);           // [NS][G][64]
            uint32_t bw[NH][2], bx[NH][2];
#pragma unroll
            for (int nh = 0; nh < NH; ++nh) {
              const int g = gid + 8 * nh;
              float w0 = 0.f, w1 = 0.f, w2 = 0.f, w3 = 0.f;
              if (g < G) {
                const unsigned char* wr = wp + (size_t)g * 256 + (rg * 16 + 2 * t4) * 4;
#pragma unroll
                for (int sx = 0; sx < CL_MAX_NS; ++sx)
                  if (sx < NS) {
                    const float ff = f[nh][sx];
                    const float2 lo = *reinterpret_cast<const float2*>(wr), hi = *reinterpret_cast<const float2*>(wr + 32);
                    w0 = fmaf(ff, lo.x, w0); w1 = fmaf(ff, lo.y, w1); w2 = fmaf(ff, hi.x, w2); w3 = fmaf(ff, hi.y, w3);
                    wr += (size_t)G * 256;
                  }
              }
              bw[nh][0] = pack2_bf16(w0, w1);
              bw[nh][1] = pack2_bf16(w2, w3);
              bx[nh][0] = split_lo(w0, w1, bw[nh][0]);
              bx[nh][1] = split_lo(w2, w3, bw[nh][1]);
            }
            const uint32_t v_u = ring_u + s * CL_TILE_BYTES;
            const uint32_t rowB = (uint32_t)((rg * 16 + lrowB) * 128);
#pragma unroll
            for (int mt = 0; mt < 8; ++mt) {
              uint32_t av[4];
              ldsm_x4_t(av, v_u + (mt >> 2) * CL_HALF + rowB + (uint32_t)(((((mt & 3) * 2 + lmid)) ^ l7) << 4));
#pragma unroll
              for (int nh = 0; nh < NH; ++nh) {
                mma_bf16_16816(yacc[mt][nh], av, bw[nh][0], bw[nh][1]);
                mma_bf16_16816(yacc[mt][nh], av, bx[nh][0], bx[nh][1]);
              }
            }
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(&bars.vempty[s]);
          s = s + CL_GROUPS < a.nV ? s + CL_GROUPS : grp;
          if (++jt == a.vt) { jt = 0; ++bl; if (t + 1 < v1) bw.next(a, pre); }
          // ---- end of the run, or of the sequence's part of it: the group's partial
          bool flush = t + 1 == v1;
          if (!flush && jt == 0) flush = bw.b != cur_b;
          if (flush) {
            const int b_ = cur_b;
            const size_t slot = (size_t)(u.h * (us.nu * P + a.B) + (w - u.h * us.nu) * P + piece + b_);
            float* red = reinterpret_cast<float*>(sm + (uint32_t)grp * 16384u);               // [4 warps][8 heads][128]
            float* ls = reinterpret_cast<float*>(sm + a.tab_off + CL_GROUPS * 512 + (uint32_t)NS * CL_ROWS * 8u) + grp * 16;   // [16] masses
            if (rg == 0 && t4 == 0) {
#pragma unroll
              for (int nh = 0; nh < NH; ++nh) {
                const int g = gid + 8 * nh;
                if (g < G) { ls[g] = l_run[nh]; a.pml[slot * G + g] = make_float2(m_run[nh], l_run[nh]); }
              }
            }
#pragma unroll
            for (int nh = 0; nh < NH; ++nh) {
              const int heads = min(8, G - nh * 8);
#pragma unroll
              for (int e = 0; e < 2; ++e) {
                const int hd = 2 * t4 + e;
                if (hd < heads) {
                  float* yp = red + (rg * 8 + hd) * D;
#pragma unroll
                  for (int mt = 0; mt < 8; ++mt) {
                    yp[mt * 16 + gid] = yacc[mt][nh][e];
                    yp[mt * 16 + gid + 8] = yacc[mt][nh][2 + e];
                  }
                }
              }
              named_barrier_sync(2 + grp, 128);
              for (int x = gt; x < heads * (D / 4); x += 128) {
                const int hd = x >> 5, c = (x & 31) * 4;
                float4 y = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int ww = 0; ww < 4; ++ww) {
                  const float4 v = *reinterpret_cast<const float4*>(red + (ww * 8 + hd) * D + c);
                  y.x += v.x; y.y += v.y; y.z += v.z; y.w += v.w;
                }
                const float l = ls[nh * 8 + hd];
                const uint2 mq = __ldg(reinterpret_cast<const uint2*>(a.mu + u.h * D + c));
                y.x = fmaf(l, __uint_as_float(mq.x << 16), y.x); y.y = fmaf(l, __uint_as_float(mq.x & 0xffff0000u), y.y);
                y.z = fmaf(l, __uint_as_float(mq.y << 16), y.z); y.w = fmaf(l, __uint_as_float(mq.y & 0xffff0000u), y.w);
                *reinterpret_cast<float4*>(a.py + (slot * G + nh * 8 + hd) * D + c) = y;
              }
              named_barrier_sync(2 + grp, 128);
            }
            if (gt == nflush++) mine = b_;
            reset();
          }
        }
        // the run's partials arrive together: one fence, an atomic per sequence, then the merges that became due
        const int expected = gt < nflush ? cl_expected(a, view, mine) : 0;
        named_barrier_sync(2 + grp, 128);
        if (gt < nflush) {
          __threadfence();                   // the partials of every thread (ordered before by the barrier) before the arrival
          if (arrive_is_last(&a.cnt[mine * a.H_kv + u.h], a.token, expected)) due[atomicAdd(ndue, 1)] = mine * a.H_kv + u.h;
          __threadfence();
        }
        named_barrier_sync(1, CL_CONS);                         // (a CTA sees a sequence become due once at most)
        cl_merge(a, view, due, *ndue, warp, CL_WARPS);
      }
    }

    if (units > 0) {                                            // the text's pieces take the memory the units' tiles were in
      if (fresh(tid) == 0) cl_text_due(a, sm)[-1] = 0;
      fence_proxy_async();
      named_barrier_sync(1, CL_CONS);
    }
    if (cl_text_part<NH>(tmKt, tmVt, a, view, sm, bars)) dead = true;
    if (dead && lane == 0) atomicExch(a.status, (int)KVC_ERR_TIMEOUT);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == CL_WARPS) tmem_dealloc(tb, 512u);
  if (NS > 1) cluster_exit_sync();
}

// ------------------------------------------------------------------------------------------ host side
template <int NH, int PL>
static const void* cluster_kernel_ptr() { return reinterpret_cast<const void*>(cluster_decode_kernel<NH, PL>); }

constexpr size_t CL_DYN_LIMIT = 231424;       // 227 KB less the barriers

// Clusters of 1 to CL_MAX_NS CTAs the device holds at once (one CTA per SM), asked once per device.  Where the query fails, clusters of that size
// are not used by the handle, and the next handle asks again: a layout and the launch that fills it always see the same answer.
void cluster_occupancy(int device, int sms, int* out) {
  static std::mutex mu;
  static int known[16][CL_MAX_NS + 1];
  std::lock_guard<std::mutex> lock(mu);
  const void* fn = cluster_kernel_ptr<1, 1>();
  out[1] = sms;
  for (int ns = 2; ns <= CL_MAX_NS; ++ns) {
    int n = device >= 0 && device < 16 ? known[device][ns] : 0;
    if (n == 0 && ensure_dynamic_smem(fn, CL_DYN_LIMIT) == cudaSuccess) {
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3((unsigned)(sms / ns * ns));
      cfg.blockDim = dim3(CL_THREADS);
      cfg.dynamicSmemBytes = CL_DYN_LIMIT;
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = (unsigned)ns; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
      cfg.attrs = attr;
      cfg.numAttrs = 1;
      if (cudaOccupancyMaxActiveClusters(&n, fn, &cfg) != cudaSuccess) { cudaGetLastError(); n = 0; }
    }
    if (n > 0 && device >= 0 && device < 16) known[device][ns] = n;
    out[ns] = n;
  }
}

// How the scores and probabilities are carried: as one bf16 term, or, where n is no multiple of 8 or a score row is too long for the
// tensor-core expansion of the three-phase kernels (which kept them in fp32 there), as two (16 bits).  The partial weights are fp32.
int cluster_terms(const kvc_layer* L) {
  const int ms = (L->mk + 15) / 16 * 16, cg = ceil_div(ms, 256);
  const bool mma = L->desc.n % 8 == 0 && expand_mma_smem_bytes(ms, (int)align_up((size_t)ceil_div(ms, cg), 16)) <= 227u * 1024u;
  return mma ? 1 : 2;
}

// CTAs a cluster has at least: at most 256 columns each, 128 where P has two terms
static int cluster_min(const kvc_layer* L) { return ceil_div(ceil_div(L->desc.n, 64), cluster_terms(L) == 2 ? 2 : 4); }

// (what decode_common's rule for the path and plan_cluster say of the handle alone)
bool cluster_may_serve(const kvc_layer* L) {
  if (L->desc.dtype != KVC_BF16 || L->passthrough || L->mode != KVC_MODE_KV || cluster_min(L) > CL_MAX_NS) return false;
  return L->use_tc == 5 || (L->use_tc == 0 && L->desc.n >= 64 && (L->desc.n % 64 == 0 || cluster_terms(L) == 2 || L->G > 1));
}

static uint32_t cl_tab_bytes(int ns) { return CL_GROUPS * 512u + (uint32_t)ns * 1024u + 256u; }
// slots of the value ring (a multiple of the groups) in ring_max bytes and the tail of the region of P
static int cl_v_slots(uint32_t ring_max, uint32_t w_bytes) {
  const int tail = (int)((CL_P_BYTES - CL_W_TAIL) / w_bytes);
  int nv = CL_V_SLOTS;
  while (nv > 0 && (uint32_t)nv * CL_TILE_BYTES + (uint32_t)(nv > tail ? nv - tail : 0) * w_bytes > ring_max) nv -= CL_GROUPS;
  return nv;
}
// Text items per (sequence, KV head): chunks of CL_TEXT_CHUNK rows, longer ones past 64 of them where the device has a warp for every
// item, past 16 where it has not.  A warp's rows are a chain of some 0.8 us per 16 of them; partials cost the merge.  4 x 2 blocks of n = 400,
// 8/2 heads, 13095 text rows: 16 items 71 us per call, 64 36.9, 128 37.1; one sequence, 32768 rows: 132, 51, 42; 2 sequences of 30000, 64/8
// heads: 154, 82, 91; more items than warps (8 sequences of 2500, 32/8 heads): 47, at 20 items 64.
static int text_items(const kvc_layer* L, int B) {
  return 64ll * B * L->desc.H_kv <= (long long)(L->num_sms > 0 ? L->num_sms : 148) * CL_WARPS ? 64 : 16;
}
static int text_chunk(const kvc_layer* L, int B, int T) {
  const int most = text_items(L, B);
  return T <= most * CL_TEXT_CHUNK ? CL_TEXT_CHUNK : (int)align_up((size_t)ceil_div(T, most), 16);
}

// Most units of a KV head and most blocks of a unit.  Uniform calls: their split.  With lengths per sequence fewer blocks than nb may split into
// more units (5 blocks into 5, but 8 into 4 of 2): clusters for all that the cap allows (else the odd ones take a second round: 38 us instead
// of 21 at 4 x 2 blocks of n = 400, 8/2 heads), of no more blocks than nb over the cap.
static UnitSplit most_units(int nb, int rbmax, int cap, bool ragged) {
  UnitSplit us = split_units(nb, rbmax, cap);
  if (!ragged || nb <= 0) return us;
  us.rb = std::min(rbmax, ceil_div(nb, cap < nb ? cap : nb));
  if (cap < nb && cap > us.nu) us.nu = cap;
  return us;
}
// expansion rows a unit of rb blocks has room for (a multiple of 8: the second term of S starts on a swizzle period)
static int unit_rows(int rb, int G) { return (int)align_up((size_t)(rb * G < CL_ROWS ? rb * G : CL_ROWS), 8); }

ClusterPlan plan_cluster(const kvc_layer* L, int B, int R, int T, bool ragged) {
  ClusterPlan p{};
  const int G = L->G, n = L->desc.n, m = L->m, H = L->desc.H_kv;
  if (L->desc.dtype != KVC_BF16 || L->passthrough || L->mode != KVC_MODE_KV || R < 1 || B < 1 || G > 16) return p;
  if (!tma_rows(L->theta_rows) || !tma_rows(L->U_rows) || (ragged && B > CL_MAX_RAGGED_B)) return p;
  if ((long long)B * R >= (1 << 28) || (long long)B * H * R >= (1ll << 31)) return p;
  p.terms = cluster_terms(L);
  p.ncg = ceil_div(n, 64);
  p.rbmax = CL_ROWS / G;
  const int nb = B * R;
  // CTAs per cluster: at most 256 columns each (128 where P has two terms); more where the smallest number of units still leaves
  // SMs to the text (the chain of a unit gets shorter), as long as every group has two slots for value tiles, whose slices of the
  // weights grow with the ranges (n = 729, 8 sequences, 28/4 heads: 6 CTAs 43.5 us, 8 CTAs with one slot per group 50.3)
  const int ns_min = cluster_min(L);
  if (ns_min > CL_MAX_NS) return p;
  const int nu_min = ceil_div(nb, p.rbmax);
  p.NS = ns_min;
  auto v_slots = [&](int ns) {
    return cl_v_slots((uint32_t)CL_DYN_LIMIT - 1024u - CL_P_BYTES - cl_tab_bytes(ns) - (ragged ? (uint32_t)(2 * B + 1) * 4u : 0u),
                      ((uint32_t)(ns * G * 256) + 127u) & ~127u);
  };
  for (int ns = p.ncg < CL_MAX_NS ? p.ncg : CL_MAX_NS; ns > ns_min; --ns)
    if ((long long)H * nu_min * 100 <= (long long)L->clusters[ns] * 87 && v_slots(ns) >= 2 * CL_GROUPS) { p.NS = ns; break; }
  p.ncl = L->clusters[p.NS];
  if (p.ncl < 1) return p;
  const double kv = 2.0 * nb * m * D * 2 * H + 4.0 * H * m * n, tx = 2.0 * B * H * (double)T * D * 2;
  p.cap = (int)(p.ncl * (kv / (kv + tx)) / H);
  if (p.cap < 1) p.cap = 1;
  {
    const int cap_max = p.ncl / H > 1 ? p.ncl / H : 1;
    p.nu_max = nu_min > cap_max ? nu_min : (cap_max < nb ? cap_max : nb);
    if (p.nu_max < 1) p.nu_max = 1;
  }
  const UnitSplit us = split_units(nb, p.rbmax, p.cap);
  const UnitSplit most = most_units(nb, p.rbmax, p.cap, ragged);
  p.ucl = (long long)H * most.nu < p.ncl ? H * most.nu : p.ncl;
  p.ms = (m + 7) & ~7;
  p.nk1 = ceil_div(m, 64);
  const int mpad = (m + 15) & ~15;
  p.npass = ceil_div(mpad, 512);
  p.prow = p.npass == 1 ? mpad : (int)align_up((size_t)ceil_div(mpad, p.npass), 64);
  p.nbox = ceil_div(p.prow, 256);
  p.brow = (int)align_up((size_t)ceil_div(p.prow, p.nbox), 16);
  if (p.npass == 1) p.prow = p.nbox * p.brow;
  p.vt = ceil_div(m, CL_TILE);
  const int planes = p.terms;
  p.srows = unit_rows(most.rb, G);
  p.s_bytes = (uint32_t)planes * p.srows * 128u;
  const uint32_t th = (uint32_t)ceil_div(p.ncg, p.NS) * 8192u, ub = (uint32_t)p.brow * 128u;
  p.x_bytes = p.s_bytes + th;
  // the A operand is read as 128 rows whatever srows is: the slot covers what the descriptor can reach
  const uint32_t reach = (uint32_t)(planes - 1) * p.srows * 128u + 16384u;
  if (p.x_bytes < reach) p.x_bytes = reach;
  if (p.x_bytes < ub) p.x_bytes = ub;
  p.x_bytes = (p.x_bytes + 1023u) & ~1023u;
  p.w_tx = (uint32_t)(p.NS * G * 256);
  p.w_bytes = (p.w_tx + 127u) & ~127u;
  const uint32_t tab = cl_tab_bytes(p.NS);
  const uint32_t pre = ragged ? (uint32_t)(2 * B + 1) * 4u : 0u;
  const uint32_t ring_max = (uint32_t)CL_DYN_LIMIT - 1024u - CL_P_BYTES - tab - pre;
  p.nK = CL_K_SLOTS;
  if ((uint32_t)p.nK * CL_TILE_BYTES > ring_max) p.nK -= CL_GROUPS;
  p.nV = cl_v_slots(ring_max, p.w_bytes);
  if (p.nV == 0) return p;
  p.nwp = (int)((CL_P_BYTES - CL_W_TAIL) / p.w_bytes) < p.nV ? (int)((CL_P_BYTES - CL_W_TAIL) / p.w_bytes) : p.nV;
  p.nX = (int)(ring_max / p.x_bytes);
  if (p.nX > CL_X_SLOTS) p.nX = CL_X_SLOTS;
  if (p.nX < 2) return p;
  p.w_off = (uint32_t)p.nV * CL_TILE_BYTES;
  uint32_t ring = (uint32_t)p.nK * CL_TILE_BYTES;
  if ((uint32_t)p.nX * p.x_bytes > ring) ring = (uint32_t)p.nX * p.x_bytes;
  if (p.w_off + (uint32_t)(p.nV - p.nwp) * p.w_bytes > ring) ring = p.w_off + (uint32_t)(p.nV - p.nwp) * p.w_bytes;
  if (ring + CL_P_BYTES < (uint32_t)CL_WARPS * CL_TEXT_SLOTS * 4096u) ring = (uint32_t)CL_WARPS * CL_TEXT_SLOTS * 4096u - CL_P_BYTES;
  ring = (ring + 127u) & ~127u;
  p.tab_off = CL_P_BYTES + ring;
  p.pre_off = p.tab_off + tab;
  p.smem = 1024u + (size_t)p.pre_off + pre;
  if (p.smem > CL_DYN_LIMIT) return p;
  p.tc = text_chunk(L, B, T);
  p.nct = ceil_div(T, p.tc);
  p.text_items = (long long)B * H * p.nct;
  if (p.text_items >= (1ll << 30)) return p;
  p.text_ded = 0;
  if (p.ucl < p.ncl && p.text_items > 0) {
    const double share = (kv + tx) * (p.ncl - p.ucl) / p.ncl / tx;
    p.text_ded = share >= 1.0 ? p.text_items : (long long)(share * p.text_items);
    // ... and at least what they can do while the units' chain runs (a unit: 18 us and 0.3 us per tile of a CTA; a warp's item: 9 us
    // with its arrival): an item behind the units ends 8-14 us after them, by the latency of one warp's pieces and merge
    const double unit_us = ceil_div(H * us.nu, p.ucl) * (18.0 + 0.3 * 2.0 * us.rb * p.vt / p.NS);
    const long long spare = (long long)(unit_us / 9.0) * (p.ncl - p.ucl) * p.NS * CL_WARPS;
    if (p.text_ded < spare) p.text_ded = spare < p.text_items ? spare : p.text_items;
    // no more clusters than the text has use for
    const long long need = (p.text_ded + (long long)p.NS * CL_WARPS - 1) / ((long long)p.NS * CL_WARPS);
    if (need < p.ncl - p.ucl) p.ncl = p.ucl + (int)need;
  } else {
    p.ncl = p.ucl;
  }
  // a CTA's list of the pairs it merges after its text items holds as many as it can have items
  const long long with = (long long)p.ucl * p.NS, without = (long long)(p.ncl - p.ucl) * p.NS;
  const long long items = std::max((p.text_items - p.text_ded + with - 1) / with, without > 0 ? (p.text_ded + without - 1) / without : 0ll);
  if (items > (long long)(CL_GROUPS * 512u + (uint32_t)p.NS * 1024u) / 4 - 1) return p;
  p.units = H * us.nu;
  p.ok = 1;
  return p;
}

// rows: of S and of the partial weights, of all clusters that take units
static ClusterWs cluster_layout(const kvc_layer* L, const ClusterPlan& p, int B, int rows) {
  ClusterWs w{};
  const int H = L->desc.H_kv, G = L->G;
  size_t off = align_up(sizeof(int) * ((size_t)B * H + 1), 256);       // behind the status word of the layout all paths share
  auto take = [&](size_t bytes) { const size_t o = off; off = align_up(off + bytes, 256); return o; };
  w.off_S = take(sizeof(__nv_bfloat16) * (size_t)rows * p.terms * p.ms);
  w.off_W = take(sizeof(float) * (size_t)rows * p.NS * p.ms);
  w.off_cnt = take(sizeof(unsigned long long) * (size_t)B * H);
  w.unit_slots = (size_t)H * ((size_t)p.nu_max * CL_GROUPS * p.NS + B);
  const size_t all = w.unit_slots + (size_t)B * H * p.nct;
  w.off_py = take(sizeof(float) * all * G * D);
  w.off_pml = take(sizeof(float2) * all * G);
  w.bytes = off;
  return w;
}
ClusterWs cluster_ws(const kvc_layer* L, const ClusterPlan& p, int B) { return cluster_layout(L, p, B, p.ucl * p.srows); }

// enough for every T <= T_cap: shorter text leaves more clusters to the units (never more than without any), which then have fewer rows each
size_t cluster_ws_bytes(const kvc_layer* L, int B, int R, int T_cap) {
  size_t most = 0;
  for (int ragged = 0; ragged < 2; ++ragged) {
    ClusterPlan p = plan_cluster(L, B, R, T_cap, ragged != 0);
    if (!p.ok) continue;
    // the chunks of a shorter text: never more than the most of a pair, nor than whole chunks of the smallest size
    p.nct = std::min(ceil_div(T_cap, CL_TEXT_CHUNK), text_items(L, B));
    const int top = plan_cluster(L, B, R, 0, ragged != 0).cap;
    int rows = 0;
    for (int cap = 1; cap <= top; ++cap) {
      const UnitSplit us = most_units(B * R, p.rbmax, cap, ragged != 0);
      rows = std::max(rows, std::min(L->desc.H_kv * us.nu, L->clusters[p.NS]) * unit_rows(us.rb, L->G));
    }
    most = std::max(most, cluster_layout(L, p, B, rows).bytes);
  }
  return most;
}

template <int NH, int PL>
static cudaError_t launch_cluster_inst(const CUtensorMap* tm, const ClusterArgs& a, const ClusterPlan& p, cudaStream_t st) {
  cudaError_t e = ensure_dynamic_smem(cluster_kernel_ptr<NH, PL>(), CL_DYN_LIMIT);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(p.ncl * p.NS));
  cfg.blockDim = dim3(CL_THREADS);
  cfg.dynamicSmemBytes = p.smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)p.NS; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = p.NS > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, cluster_decode_kernel<NH, PL>, tm[0], tm[1], tm[2], tm[3], tm[4], tm[5], tm[6], tm[7], tm[8], a);
}

cudaError_t launch_cluster(const kvc_layer* L, const DecodeArgs& d, const ClusterPlan& p, char* ws, cudaStream_t st, bool* encoded) {
  *encoded = false;
  const int B = d.B, H = d.H_kv, R = d.R, G = d.G, m = L->m, n = L->desc.n;
  const ClusterWs w = cluster_ws(L, p, B);
  const int planes = p.terms;
  CUtensorMap tm[9];
  {
    // capsule rows as (64 channels, m rows of a block, channel half, blocks): a box lands as [half][64 rows][64]
    const uint64_t dims[4] = {64ull, (uint64_t)m, 2ull, (uint64_t)B * H * R};
    const uint64_t str[3] = {256ull, 128ull, (uint64_t)m * 256};
    const uint32_t box[4] = {64u, (uint32_t)CL_TILE, 2u, 1u};
    if (!encode_tensor_map_bf16(&tm[0], d.Kc, 4, dims, str, box) || !encode_tensor_map_bf16(&tm[1], d.Vc, 4, dims, str, box)) return cudaSuccess;
  }
  if (d.T > 0) {
    const uint64_t dims[5] = {64ull, (uint64_t)d.T, 2ull, (uint64_t)H, (uint64_t)B};
    const uint64_t str[4] = {256ull, 128ull, (uint64_t)d.T_cap * 256, (uint64_t)H * d.T_cap * 256};
    const uint32_t box[5] = {64u, 16u, 2u, 1u, 1u};
    if (!encode_tensor_map_bf16(&tm[2], d.K_txt, 5, dims, str, box) || !encode_tensor_map_bf16(&tm[3], d.V_txt, 5, dims, str, box)) return cudaSuccess;
  } else {
    tm[2] = tm[0];
    tm[3] = tm[0];
  }
  {
    const uint64_t dims[4] = {(uint64_t)m, (uint64_t)p.srows, (uint64_t)planes, (uint64_t)p.ucl};
    const uint64_t str[3] = {(uint64_t)p.ms * 2, (uint64_t)p.srows * p.ms * 2, (uint64_t)planes * p.srows * p.ms * 2};
    const uint32_t box[4] = {64u, (uint32_t)p.srows, (uint32_t)planes, 1u};
    if (!encode_tensor_map_bf16(&tm[4], ws + w.off_S, 4, dims, str, box)) return cudaSuccess;
  }
  for (int x = 0; x < 2; ++x) {
    // theta as (64 columns, m rows, 64-column groups, H_kv): a box lands as [group][64 rows][64]; boxes of ceil and floor(ncg / NS)
    const int groups = x == 0 ? ceil_div(p.ncg, p.NS) : (p.ncg / p.NS > 0 ? p.ncg / p.NS : 1);
    const uint64_t dims[4] = {64ull, (uint64_t)m, (uint64_t)p.ncg, (uint64_t)H};
    const uint64_t str[3] = {(uint64_t)L->theta_np * 2, 128ull, (uint64_t)m * L->theta_np * 2};
    const uint32_t box[4] = {64u, 64u, (uint32_t)groups, 1u};
    if (!encode_tensor_map_bf16(&tm[5 + x], L->theta_rows, 4, dims, str, box)) return cudaSuccess;
  }
  {
    const uint64_t dims[3] = {(uint64_t)n, (uint64_t)m, (uint64_t)H};           // columns past n are zero-filled
    const uint64_t str[2] = {(uint64_t)L->U_np * 2, (uint64_t)m * L->U_np * 2};
    const uint32_t box[3] = {64u, (uint32_t)p.brow, 1u};
    if (!encode_tensor_map_bf16(&tm[7], L->U_rows, 3, dims, str, box)) return cudaSuccess;
  }
  {
    const uint64_t dims[4] = {(uint64_t)p.ms, (uint64_t)p.srows, (uint64_t)p.NS, (uint64_t)p.ucl};
    const uint64_t str[3] = {(uint64_t)p.ms * 4, (uint64_t)p.srows * p.ms * 4, (uint64_t)p.NS * p.srows * p.ms * 4};
    const uint32_t box_ld[4] = {64u, (uint32_t)G, (uint32_t)p.NS, 1u};
    const bool ok = encode_tensor_map_f32(&tm[8], ws + w.off_W, 4, dims, str, box_ld, false);
    if (!ok) return cudaSuccess;
  }
  *encoded = true;
  ClusterArgs a{};
  a.q = static_cast<const __nv_bfloat16*>(d.q);
  a.mu = static_cast<const __nv_bfloat16*>(d.mu);
  a.Kc = static_cast<const __nv_bfloat16*>(d.Kc); a.Vc = static_cast<const __nv_bfloat16*>(d.Vc);
  a.theta = static_cast<const __nv_bfloat16*>(L->theta_rows); a.U = static_cast<const __nv_bfloat16*>(L->U_rows);
  a.theta_np = L->theta_np; a.U_np = L->U_np;
  a.out = static_cast<__nv_bfloat16*>(d.out);
  a.S = reinterpret_cast<__nv_bfloat16*>(ws + w.off_S);
  a.W = reinterpret_cast<float*>(ws + w.off_W);
  a.py = reinterpret_cast<float*>(ws + w.off_py);
  a.pml = reinterpret_cast<float2*>(ws + w.off_pml);
  a.tslot0 = (int)w.unit_slots;
  a.cnt = reinterpret_cast<unsigned long long*>(ws + w.off_cnt);
  a.token = d.token; a.status = d.status; a.R_b = d.R_b; a.T_b = d.T_b; a.early = d.early_capsules;
  a.B = B; a.H_kv = H; a.G = G; a.R = R; a.m = m; a.n = n; a.T = d.T;
  a.NS = p.NS; a.ncl = p.ncl; a.ucl = p.ucl; a.cap = p.cap; a.rbmax = p.rbmax; a.ncg = p.ncg; a.ms = p.ms; a.nk1 = p.nk1;
  a.npass = p.npass; a.prow = p.prow; a.nbox = p.nbox; a.brow = p.brow; a.vt = p.vt; a.srows = p.srows; a.nK = p.nK; a.nX = p.nX; a.nV = p.nV;
  a.x_bytes = p.x_bytes; a.s_bytes = p.s_bytes; a.w_off = p.w_off; a.w_bytes = p.w_bytes; a.w_tx = p.w_tx; a.nwp = p.nwp;
  a.tab_off = p.tab_off; a.pre_off = p.pre_off;
  a.tc = p.tc; a.nct = p.nct; a.text_items = (int)p.text_items; a.text_ded = (int)p.text_ded;
  ProfScope prof(KVC_KERNEL_FUSED, st, KVC_KERNEL_CLUSTER);
  if (G > 8)
    return p.terms == 1 ? launch_cluster_inst<2, 1>(tm, a, p, st) : launch_cluster_inst<2, 2>(tm, a, p, st);
  return p.terms == 1 ? launch_cluster_inst<1, 1>(tm, a, p, st) : launch_cluster_inst<1, 2>(tm, a, p, st);
}

}  // namespace kvc
