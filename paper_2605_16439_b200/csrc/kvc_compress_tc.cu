// Prefill compression of bf16 storage in one kernel (Sec. 3.2 "Prefilling Stage"): for every block a sequence has, the
// retained key rows (C2) and V_tilde = U[h] (V - 1 mu[h]^T) (C3), taken as  U V - (U 1) mu^T  with the row sums of U computed
// once per layer; for batches with per-sequence lengths also the lengths themselves and the rows left over.
//
// Bound: HBM (the retained key rows in and out, V in, V_tilde out), with the projection's operands streamed through shared
// memory beside it.  One persistent CTA per SM:
//   warps 0-7       epilogue: one lane per output row and half of the channels each; minus usum[j] mu[c], rounded to bf16,
//                   turned through shared memory so that a store covers four rows of 128 bytes
//   warp 8          MMA issue: tcgen05.mma M = 128, N = 256, K = 16; a 128-row tile of U is the K-major A operand, the V rows of
//                   two blocks (channels contiguous) the MN-major B operand, read as the TMA engine laid them down.  A unit
//                   (row tile, pair of blocks) fills 256 tensor-memory columns; there are two such sets, so a unit's epilogue
//                   (about 3.6 k cycles) runs behind the next unit's products
//   warp 9          TMA producer: per 64 vision positions one 48 KB stage (U 16 KB, V 2 x 16 KB, 128-byte swizzle), a ring of
//                   stages that runs on across units
//   warps 10-15     row copies: the retained key rows, a side stored verbatim, the rows left over by a ragged batch
// Measured on B200 (per layer, back to back): 8 x 32 x 5 blocks of n = 576, m = 231: 84 us (5.1 TB/s of 426 MB; 129 us with one
// launch for the keys and one CTA per (block, row tile)); 8 sequences of up to 8 blocks x 4 heads of n = 1024, m = 410 with their
// own lengths: 42 us (1108 us on the CUDA cores before).  Tried: both row tiles of a pair in one unit, which fills the tensor memory
// and leaves the epilogue exposed (N = 256: 103 us at the first shape; N = 128: 94 us).
// Any n: the tensor maps clip the last stage of a block (U is read from the layer's copy with a 16-byte row pitch where its own
// rows are not aligned), so block lengths that are no multiple of 64 and ragged batches take the same kernel.
#include "kvc_tma.cuh"
#include "kvc_tcgen05.cuh"
#include "kvc_internal.cuh"

namespace kvc {

constexpr int CT_MAX_STAGES = 4;
constexpr int CT_BM = 128, CT_BK = 64;
constexpr uint32_t CT_U_BYTES = CT_BM * CT_BK * 2;          // 16 KB: one row tile of U, 64 columns
constexpr uint32_t CT_V_BYTES = CT_BK * D * 2;              // 16 KB: 64 rows of V as two 64-channel halves
constexpr int CT_EPI_WARPS = 8;
constexpr uint32_t CT_OUT_WARP = 32 * 128;                  // epilogue staging of a warp: 32 rows, one 64-channel half
constexpr uint32_t CT_TMEM_COLS = 512;
// Six: sixteen warps have 128 registers a thread; with eight (96 registers) the copy loop's two steps in flight spilled, an L2 round trip
// each with the L1 given to shared memory (one layer's buffers again and again: 8 x 5 blocks of n = 576, 32 heads, ratio 0.6: 78 us, six 74.5; 32 x 8 of 256: 31 and 27)
constexpr int CT_COPY_WARPS = 6;
constexpr int CT_THREADS = (CT_EPI_WARPS + 2 + CT_COPY_WARPS) * 32;
constexpr uint32_t CT_SMEM_LIMIT = 231424;                  // dynamic part of the 227 KB; the barriers take the rest
constexpr int CT_MAX_B = 8192;                              // sequences of a ragged batch: their block counts sit in shared memory

// rows copied per block of a (sequence, KV head): source row idx[h][j] (or j), destination row j
struct CopySide {
  const __nv_bfloat16* src;
  __nv_bfloat16* dst;
  const int32_t* idx;        // [H_kv][rows], nullptr: the first `rows` rows of the block
  int rows;                  // 0: nothing to copy on this side
};

struct CompressTcArgs {
  CopySide copy[2];          // keys, values
  __nv_bfloat16* Vc;         // [B*H_kv*R][m][D]
  const float* usum;         // [H_kv][m] row sums of U
  const __nv_bfloat16* mu;   // [H_kv][D]
  int project;               // 1: values are projected
  int B, H_kv, R, n, m;
  int bpu;                   // a unit: one 128-row tile of U and `bpu` blocks (1 or 2)
  int mtiles;                // row tiles of U
  int stages;
  uint32_t stage_bytes;
  long long pitch;           // vision rows per (sequence, KV head) of the source
  // per-sequence lengths (nullptr: R blocks each)
  const int* N_v;
  int N_cap, T_cap;
  int* R_b;                  // written by CTA 0 (nullptr: not at all)
  int* T_b;
  const __nv_bfloat16* Ktail_src;
  const __nv_bfloat16* Vtail_src;
  __nv_bfloat16* K_tail;
  __nv_bfloat16* V_tail;
  int* status;
};

// block count and rows left over of a sequence with nv vision rows; false if a length did not fit and was clamped
__device__ __forceinline__ bool ragged_split(int nv, const CompressTcArgs& a, int& r, int& t) {
  bool ok = nv >= 0 && nv <= a.N_cap;
  nv = nv < 0 ? 0 : (nv > a.N_cap ? a.N_cap : nv);
  r = nv / a.n;
  t = nv - r * a.n;
  if (r > a.R) { ok = false; r = a.R; t = 0; }
  if (t > a.T_cap) { ok = false; t = a.T_cap; }
  return ok;
}

struct BlockList {                 // the blocks of one KV head in (sequence, block) order
  const int* pre;                  // prefix sums of the block counts, nullptr: R blocks per sequence
  int B, R;
  __device__ __forceinline__ int total() const { return pre ? pre[B] : B * R; }
  __device__ __forceinline__ void locate(int k, int& b, int& r) const {
    if (!pre) { b = k / R; r = k - b * R; return; }
    int lo = 0, hi = B;            // pre[lo] <= k < pre[hi]
    while (hi - lo > 1) { const int mid = (lo + hi) >> 1; if (pre[mid] <= k) lo = mid; else hi = mid; }
    b = lo; r = k - pre[lo];
  }
};

__device__ __forceinline__ uint4 ld_stream(const void* p) {
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];\n" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}

// one step of a row copy: up to 16 rows of a block
struct CopyStep {
  const __nv_bfloat16* src;        // row 0 of the block, this lane's 16-byte column
  __nv_bfloat16* dst;              // destination row j0
  int row;                         // lane x, x + 16: source row of the step's row x (row 0 past the last one)
  int rows;                        // rows of the step, possibly none
};

__global__ void __launch_bounds__(CT_THREADS, 1)
compress_kernel(const __grid_constant__ CUtensorMap tmU, const __grid_constant__ CUtensorMap tmV, const CompressTcArgs a) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* sm = smem_raw + ((1024u - (smem_addr(smem_raw) & 1023u)) & 1023u);
  __shared__ __align__(8) uint64_t full_bar[CT_MAX_STAGES], empty_bar[CT_MAX_STAGES], acc_full[2], acc_free[2];
  __shared__ uint32_t s_tmem;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  unsigned char* staging = sm + (uint32_t)a.stages * a.stage_bytes;
  __nv_bfloat16* s_mu = reinterpret_cast<__nv_bfloat16*>(staging + CT_EPI_WARPS * CT_OUT_WARP);     // [epilogue warps][64]
  int* s_pre = reinterpret_cast<int*>(s_mu + CT_EPI_WARPS * 64);                                    // [B + 1] (ragged batches)

  if (tid == 0) {
    for (int s = 0; s < a.stages; ++s) { mbar_init(&full_bar[s], 1); mbar_init(&empty_bar[s], 1); }
    for (int x = 0; x < 2; ++x) { mbar_init(&acc_full[x], 1); mbar_init(&acc_free[x], CT_EPI_WARPS); }
    fence_mbar_init();
  }
  if (warp == CT_EPI_WARPS && a.project) tmem_alloc(&s_tmem, CT_TMEM_COLS);
  grid_dep_wait();
  grid_dep_launch();
  // the status word of this call: only CTA 0 reports lengths, after clearing it; a bounded wait gives up after a second
  if (blockIdx.x == 0 && tid == 0) *a.status = 0;
  if (a.N_v && warp == 0) {
    __syncwarp();
    // block counts -> prefix sums, 32 sequences at a time
    int carry = 0;
    if (lane == 0) s_pre[0] = 0;
    for (int b0 = 0; b0 < a.B; b0 += 32) {
      const int b = b0 + lane;
      int r = 0, t = 0;
      bool ok = true;
      if (b < a.B) ok = ragged_split(a.N_v[b], a, r, t);
      if (b < a.B && blockIdx.x == 0) {
        if (a.R_b) { a.R_b[b] = r; a.T_b[b] = t; }
        if (!ok) atomicExch(a.status, (int)KVC_ERR_BOUNDS);
      }
      int x = r;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) { const int y = __shfl_up_sync(0xffffffffu, x, o); if (lane >= o) x += y; }
      if (b < a.B) s_pre[b + 1] = carry + x;
      carry += __shfl_sync(0xffffffffu, x, 31);
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const BlockList list{a.N_v ? s_pre : nullptr, a.B, a.R};
  const int nblk = list.total();                                    // blocks of one KV head
  const int nk = (a.n + CT_BK - 1) / CT_BK;
  const int nbp = (nblk + a.bpu - 1) / a.bpu;
  const int units = a.project ? a.H_kv * nbp * a.mtiles : 0;       // unit = ((h * nbp) + k) * mtiles + tile
  auto unit_of = [&](int u, int& h, int& k0, int& row0) {
    const int hk = u / a.mtiles;
    row0 = (u - hk * a.mtiles) * CT_BM;
    h = hk / nbp;
    k0 = (hk - h * nbp) * a.bpu;
  };

  if (warp >= CT_EPI_WARPS + 2) {
    // ---------------- row copies: a contiguous run of 16-row steps per warp, the next step's eight 16-byte loads per lane
    // (and the indices of the one after it) in flight while a step is stored ----------------
    const int cw = blockIdx.x * CT_COPY_WARPS + (warp - CT_EPI_WARPS - 2), ncw = gridDim.x * CT_COPY_WARPS;
    const int sub = lane >> 4, c = lane & 15;
    // jobs: 0 keys, 1 values (a side stored verbatim), 2 the rows left over by a ragged batch
    for (int job = 0; job < 3; ++job) {
      const bool tail = job == 2;
      if (tail ? !(a.N_v && a.T_cap > 0) : a.copy[job].rows == 0) continue;
      const int rows = tail ? a.n : a.copy[job].rows;
      const int cpb = (rows + 15) >> 4;
      const long long chunks = (tail ? 2ll * a.B * a.H_kv : (long long)a.H_kv * nblk) * cpb;
      const long long c0 = chunks * cw / ncw, c1 = chunks * (cw + 1) / ncw;
      if (c0 >= c1) continue;
      int hk = (int)(c0 / cpb), jc = (int)(c0 - (long long)hk * cpb);
      const __nv_bfloat16 *src = nullptr;
      __nv_bfloat16* dst = nullptr;
      const int32_t* idx = nullptr;
      int limit = 0;
      auto locate = [&]() {                      // the block (or the rows left over) number hk
        if (tail) {
          const int side = hk & 1, pair = hk >> 1;
          int r, t;
          ragged_split(a.N_v[pair / a.H_kv], a, r, t);
          limit = t;
          src = (side ? a.Vtail_src : a.Ktail_src) + ((long long)pair * a.pitch + (long long)r * a.n) * D + c * 8;
          dst = (side ? a.V_tail : a.K_tail) + (long long)pair * a.T_cap * D + c * 8;
        } else {
          const CopySide& s = a.copy[job];
          const int h = hk / nblk;
          int b, r;
          list.locate(hk - h * nblk, b, r);
          const long long pair = (long long)b * a.H_kv + h;
          limit = rows;
          idx = s.idx ? s.idx + (size_t)h * rows : nullptr;
          src = s.src + (pair * a.pitch + (long long)r * a.n) * D + c * 8;
          dst = s.dst + ((pair * a.R + r) * rows) * D + c * 8;
        }
      };
      locate();
      auto next_step = [&]() {                   // describes the current step and moves on
        CopyStep st;
        st.src = src;
        st.dst = dst + (size_t)jc * 16 * D;
        const int j = jc * 16 + c;
        st.rows = limit - jc * 16;
        st.row = j < limit ? (idx ? __ldg(idx + j) : j) : 0;
        if (++jc == cpb) { jc = 0; ++hk; if (hk * (long long)cpb < c1) locate(); }
        return st;
      };
      auto load = [&](const CopyStep& st, uint4 (&v)[8]) {
        if (st.rows <= 0) return;
#pragma unroll
        for (int x = 0; x < 8; ++x) v[x] = ld_stream(st.src + (size_t)__shfl_sync(0xffffffffu, st.row, 2 * x + sub) * D);
      };
      auto store = [&](const CopyStep& st, const uint4 (&v)[8]) {
#pragma unroll
        for (int x = 0; x < 8; ++x)
          if (2 * x + sub < st.rows) *reinterpret_cast<uint4*>(st.dst + (size_t)(2 * x + sub) * D) = v[x];
      };
      const int steps = (int)(c1 - c0);
      uint4 va[8], vb[8];
      CopyStep sa = next_step(), sb = sa;
      load(sa, va);
      if (steps > 1) sb = next_step();
      for (int it = 0; it < steps; it += 2) {
        CopyStep sc = sb;
        if (it + 1 < steps) load(sb, vb);
        if (it + 2 < steps) sc = next_step();
        store(sa, va);
        if (it + 1 < steps) {
          if (it + 2 < steps) load(sc, va);
          CopyStep sd = sc;
          if (it + 3 < steps) sd = next_step();
          store(sb, vb);
          sa = sc;
          sb = sd;
        }
      }
    }
  } else if (warp == CT_EPI_WARPS + 1) {
    // ---------------- producer ----------------
    if (lane == 0 && units > 0) {
      tma_prefetch_desc(&tmU); tma_prefetch_desc(&tmV);
      uint32_t slot = 0, phase = 1;
      bool ok = true;
      for (int u = blockIdx.x; u < units && ok; u += gridDim.x) {
        int h, k0, row0, b[2], r[2];
        unit_of(u, h, k0, row0);
        const int nb = min(a.bpu, nblk - k0);
        list.locate(k0, b[0], r[0]);
        if (nb > 1) list.locate(k0 + 1, b[1], r[1]);
        int kc = u % nk;                         // CTAs that share U[h] walk its columns from different starts
        for (int i = 0; i < nk; ++i, kc = kc + 1 < nk ? kc + 1 : 0) {
          if (!mbar_wait_bounded(&empty_bar[slot], phase)) { ok = false; break; }
          unsigned char* dst = sm + slot * a.stage_bytes;
          mbar_expect_tx(&full_bar[slot], (uint32_t)nb * CT_V_BYTES + CT_U_BYTES);
          for (int x = 0; x < nb; ++x)
            tma_load_5d(dst + x * CT_V_BYTES, &tmV, 0, kc * CT_BK, 0, x ? r[1] : r[0], (x ? b[1] : b[0]) * a.H_kv + h, &full_bar[slot]);
          tma_load_3d(dst + a.bpu * CT_V_BYTES, &tmU, kc * CT_BK, row0, h, &full_bar[slot]);
          if (++slot == (uint32_t)a.stages) { slot = 0; phase ^= 1u; }
        }
      }
      if (!ok) atomicExch(a.status, (int)KVC_ERR_TIMEOUT);
    }
  } else if (warp == CT_EPI_WARPS) {
    // ---------------- MMA issue: a unit accumulates in columns [256 set, + 128 blocks) ----------------
    const uint32_t tb = s_tmem;
    const uint32_t v_off = (uint32_t)a.bpu * CT_V_BYTES;
    // descriptors of the ring's first stage; a stage, a tile of U and a K step advance the address field
    const uint64_t adesc0 = umma_smem_desc(smem_addr(sm) + v_off, 16u, 1024u, UMMA_LAYOUT_SW128);
    const uint64_t bdesc0 = umma_smem_desc(smem_addr(sm), CT_V_BYTES / 2, 1024u, UMMA_LAYOUT_SW128);
    uint32_t slot = 0, phase = 0, acc = 0, acc_phase = 1;
    bool dead = false;
    for (int u = blockIdx.x; u < units; u += gridDim.x) {
      int h, k0, row0;
      unit_of(u, h, k0, row0);
      const int nb = min(a.bpu, nblk - k0);
      const uint32_t idesc = umma_idesc_bf16(128, 128 * nb, 0, 1);
      if (!dead && !mbar_wait_bounded(&acc_free[acc], acc_phase)) dead = true;
      __syncwarp();
      tc_fence_after();
      for (int kc = 0; kc < nk; ++kc) {
        if (!dead && !mbar_wait_bounded(&full_bar[slot], phase)) dead = true;
        __syncwarp();
        tc_fence_after();
        if (lane == 0 && !dead) {
          const uint64_t ad = adesc0 + (uint64_t)((slot * a.stage_bytes) >> 4), bd = bdesc0 + (uint64_t)((slot * a.stage_bytes) >> 4);
          const uint32_t d0 = tb + acc * 256u;
#pragma unroll
          for (int ks = 0; ks < 4; ++ks) umma_bf16(d0, ad + (uint64_t)(ks * 2), bd + (uint64_t)(ks * 128), idesc, (kc | ks) ? 1u : 0u);
          umma_commit(&empty_bar[slot]);
          if (kc == nk - 1) umma_commit(&acc_full[acc]);
        }
        __syncwarp();
        if (++slot == (uint32_t)a.stages) { slot = 0; phase ^= 1u; }
      }
      acc ^= 1u;
      if (acc == 0) acc_phase ^= 1u;
    }
    if (dead && lane == 0) atomicExch(a.status, (int)KVC_ERR_TIMEOUT);
  } else {
    // ---------------- epilogue: V_tilde[j][c] = acc - usum[j] mu[c]; a warp has a lane quarter and one 64-channel half ----------------
    const int qw = warp & 3, hf = warp >> 2;
    const uint32_t tb = s_tmem + ((uint32_t)(qw * 32) << 16);
    unsigned char* out_sm = staging + (uint32_t)warp * CT_OUT_WARP;
    uint32_t acc = 0, phase = 0;
    int cur_h = -1;
    __nv_bfloat16* mu = s_mu + warp * 64;         // this half's channels of mu[h]
    bool ok = true;
    for (int u = blockIdx.x; u < units; u += gridDim.x) {
      int h, k0, row0;
      unit_of(u, h, k0, row0);
      const int nb = min(a.bpu, nblk - k0);
      if (h != cur_h) {
        cur_h = h;
        __syncwarp();
        *reinterpret_cast<uint32_t*>(mu + lane * 2) = *reinterpret_cast<const uint32_t*>(a.mu + h * D + hf * 64 + lane * 2);
        __syncwarp();
      }
      const int j0 = row0 + qw * 32;
      const float us = j0 + lane < a.m ? __ldg(a.usum + (size_t)h * a.m + j0 + lane) : 0.f;
      if (ok && !mbar_wait_bounded(&acc_full[acc], phase)) ok = false;
      __syncwarp();
      tc_fence_after();
      for (int x = 0; x < nb; ++x) {
        int b, r;
        list.locate(k0 + x, b, r);
        const int bhr = (b * a.H_kv + h) * a.R + r;
        if (j0 >= a.m) break;
        const uint32_t col = tb + acc * 256u + (uint32_t)(x * 128 + hf * 64);
#pragma unroll
        for (int c0 = 0; c0 < 2; ++c0) {
          uint32_t v[32];
          tmem_ld_issue_x32(col + (uint32_t)(c0 * 32), v);
          tmem_ld_wait_x32(v);
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            uint32_t w[4];
            const uint4 m4 = *reinterpret_cast<const uint4*>(mu + c0 * 32 + q * 8);
            const uint32_t mq[4] = {m4.x, m4.y, m4.z, m4.w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const uint32_t mm = mq[k];
              w[k] = pack2_bf16(fmaf(-us, __uint_as_float(mm << 16), __uint_as_float(v[8 * q + 2 * k])),
                                fmaf(-us, __uint_as_float(mm & 0xffff0000u), __uint_as_float(v[8 * q + 2 * k + 1])));
            }
            *reinterpret_cast<uint4*>(out_sm + swz(lane, c0 * 4 + q)) = make_uint4(w[0], w[1], w[2], w[3]);
          }
        }
        __syncwarp();
        // four rows of 128 bytes per store instruction
        __nv_bfloat16* dst = a.Vc + ((size_t)bhr * a.m + j0) * D + hf * 64 + (lane & 7) * 8;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const int rr = q * 4 + (lane >> 3);
          const uint4 w = *reinterpret_cast<const uint4*>(out_sm + swz(rr, lane & 7));
          if (ok && j0 + rr < a.m) *reinterpret_cast<uint4*>(dst + (size_t)rr * D) = w;
        }
        __syncwarp();
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&acc_free[acc]);
      acc ^= 1u;
      if (acc == 0) phase ^= 1u;
    }
    if (!ok && lane == 0) atomicExch(a.status, (int)KVC_ERR_TIMEOUT);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == CT_EPI_WARPS && a.project) tmem_dealloc(s_tmem, CT_TMEM_COLS);
}

// bf16 storage, 16-byte aligned pointers.  N_v == nullptr: a uniform batch of R blocks per sequence (pitch R n); otherwise
// per-sequence lengths.  keys / values say what happens on a side: 0 nothing, 1 the method (retained rows / projection),
// 2 copied verbatim.  *used == false (and nothing launched) if this kernel does not apply.
cudaError_t launch_compress_tc(const kvc_layer* L, const void* K_vis, const void* V_vis, int B, int R, long long pitch, int keys,
                               int values, void* Kc, void* Vc, const RaggedCompress* rag, cudaStream_t st, bool* used) {
  *used = false;
  const int n = L->desc.n, m = L->m, H_kv = L->desc.H_kv;
  if (L->desc.dtype != KVC_BF16) return cudaSuccess;
  uintptr_t align = reinterpret_cast<uintptr_t>(K_vis) | reinterpret_cast<uintptr_t>(V_vis) | reinterpret_cast<uintptr_t>(Kc) |
                    reinterpret_cast<uintptr_t>(Vc);
  if (rag) align |= reinterpret_cast<uintptr_t>(rag->K_tail) | reinterpret_cast<uintptr_t>(rag->V_tail);
  if (align & 15) return cudaSuccess;
  if (rag && B > CT_MAX_B) return cudaSuccess;
  if ((long long)B * H_kv * R >= (1ll << 31) || (long long)B * R >= (1ll << 30)) return cudaSuccess;
  CompressTcArgs a{};
  CUtensorMap tmU{}, tmV{};
  const bool project = values == 1 && R > 0;
  if (project) {
    if ((reinterpret_cast<uintptr_t>(L->desc.mu) & 7) || !L->d_usum || !tma_rows(L->U_rows)) return cudaSuccess;
    {
      const uint64_t dims[3] = {(uint64_t)n, (uint64_t)m, (uint64_t)H_kv};
      const uint64_t str[2] = {(uint64_t)L->U_np * 2, (uint64_t)m * L->U_np * 2};
      const uint32_t box[3] = {64u, (uint32_t)CT_BM, 1u};
      if (!encode_tensor_map_bf16(&tmU, L->U_rows, 3, dims, str, box)) return cudaSuccess;
    }
    {
      // V as (64 channels, n rows of a block, channel half, blocks, pairs): a box lands as [half][64 rows][64], rows past the
      // block's last are zero-filled
      const long long rb = pitch / n < R ? pitch / n : R;
      const uint64_t dims[5] = {64ull, (uint64_t)n, 2ull, (uint64_t)(rb < 1 ? 1 : rb), (uint64_t)B * H_kv};
      const uint64_t str[4] = {256ull, 128ull, (uint64_t)n * 256, (uint64_t)pitch * 256};
      const uint32_t box[5] = {64u, (uint32_t)CT_BK, 2u, 1u, 1u};
      if (!encode_tensor_map_bf16(&tmV, V_vis, 5, dims, str, box)) return cudaSuccess;
    }
  }
  a.project = project ? 1 : 0;
  a.copy[0].src = static_cast<const __nv_bfloat16*>(K_vis); a.copy[0].dst = static_cast<__nv_bfloat16*>(Kc);
  a.copy[0].idx = keys == 1 ? L->d_idx : nullptr; a.copy[0].rows = keys && R > 0 ? L->mk : 0;
  a.copy[1].src = static_cast<const __nv_bfloat16*>(V_vis); a.copy[1].dst = static_cast<__nv_bfloat16*>(Vc);
  a.copy[1].idx = nullptr; a.copy[1].rows = values == 2 && R > 0 ? L->mv : 0;
  a.Vc = static_cast<__nv_bfloat16*>(Vc);
  a.usum = L->d_usum;
  a.mu = static_cast<const __nv_bfloat16*>(L->desc.mu);
  a.B = B; a.H_kv = H_kv; a.R = R; a.n = n; a.m = m; a.pitch = pitch;
  const long long blocks = (long long)B * H_kv * R;
  const int sms = L->num_sms > 0 ? L->num_sms : 148;
  // Two blocks per unit give the MMA its full width of 256 columns (141 cycles per K step of 16 against 95 for half the width); one
  // where those units are no more than the SMs (2 x 3 blocks of n = 576, m = 288, 8 heads: 9.4 us, in pairs 10.3), since a second wave of
  // them costs more than the width (3 x 3: 13.5 and 10.9; 2 x 5 of 1024, m = 410, 4 heads: 18.8 and 13.6).
  a.bpu = 1;
  a.mtiles = ceil_div(m, CT_BM);
  auto unit_count = [&]() { return ((long long)B * R + a.bpu - 1) / a.bpu * H_kv * a.mtiles; };
  if (unit_count() > sms) a.bpu = 2;
  if (unit_count() >= (1ll << 31)) return cudaSuccess;
  *used = true;
  a.status = L->d_cstatus;
  if (rag) {
    a.N_v = rag->N_v; a.N_cap = rag->N_cap; a.T_cap = rag->T_cap; a.R_b = rag->R_b; a.T_b = rag->T_b;
    a.Ktail_src = static_cast<const __nv_bfloat16*>(K_vis); a.Vtail_src = static_cast<const __nv_bfloat16*>(V_vis);
    a.K_tail = static_cast<__nv_bfloat16*>(rag->K_tail); a.V_tail = static_cast<__nv_bfloat16*>(rag->V_tail);
  }
  a.stage_bytes = CT_U_BYTES + (uint32_t)a.bpu * CT_V_BYTES;
  const size_t fixed = CT_EPI_WARPS * CT_OUT_WARP + CT_EPI_WARPS * 128 + (rag ? sizeof(int) * ((size_t)B + 1) : 0) + 1024;
  a.stages = (int)((CT_SMEM_LIMIT - fixed) / a.stage_bytes);
  if (a.stages > CT_MAX_STAGES) a.stages = CT_MAX_STAGES;
  const size_t smem = (size_t)a.stages * a.stage_bytes + fixed;
  cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(compress_kernel), smem);
  if (e != cudaSuccess) return e;
  ProfScope prof(project ? KVC_KERNEL_PROJECT_VALUES : KVC_KERNEL_GATHER_KEYS, st, KVC_KERNEL_COMPRESS);
  long long grid = project ? unit_count() : 1;
  for (int s = 0; s < 2; ++s) {
    const long long c = (blocks * ceil_div(a.copy[s].rows, 16) + CT_COPY_WARPS - 1) / CT_COPY_WARPS;
    grid = c > grid ? c : grid;
  }
  if (rag) {
    const long long c = (2ll * B * H_kv * ceil_div(n, 16) + CT_COPY_WARPS - 1) / CT_COPY_WARPS;
    grid = c > grid ? c : grid;
  }
  return launch_dependent(compress_kernel, dim3((unsigned)(grid < sms ? grid : sms)), dim3(CT_THREADS), smem, st, tmU, tmV, a);
}

}  // namespace kvc
