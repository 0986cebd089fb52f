// Steps 2 and 3 of Algorithm 1 for one KV head: L_img = S_full theta, P = exp(L_img - rowmax),
// W = P U^T.  Rows are the (sequence, query head in group, block) triples that share theta[h] and
// U[h]; every row keeps its own running maximum (the joint softmax over all blocks and the text is
// completed by the log-sum-exp merge of the output kernel), and the n axis may be split over
// several CTAs, each emitting an unnormalised partial (W, max, sum).
//
// This translation unit holds the CUDA-core fp32 version, used for fp32 storage (1e-4 parity) and
// as the fallback shape-agnostic path.  It also serves the one-sided variants (App. G): with verbatim
// keys the score row already has n entries and the expansion is the identity (id_theta); with verbatim
// values the weight row has n entries and equals P (id_U).  The score row has a.m entries (pitch a.ms),
// the weight row a.mv entries (pitch a.msv).
#include "kvc_async.cuh"
#include "kvc_internal.cuh"

namespace kvc {

// Bound: latency of the parameter loads from L2 at the few rows this path is used for, fp32 multiply-adds beyond.  A CTA has 16 rows and
// walks its range of the n axis in chunks of 64 positions:
//   L      thread <-> (position, quarter of the retained rows), eight loads of theta in flight, 16 rows accumulated in registers
//          against scores broadcast from shared memory ([j][16 rows]); the quarters meet in shared memory
//   W      thread <-> a row of U (and every 256th after it), 16-byte loads of its 64 entries, the probabilities broadcast; in bf16,
//          rows that do not start on 16-byte boundaries, or at most 64 of them, 64 at a time through shared memory, thread <-> (row, 4
//          expansion rows)
//          (32 sequences of one block of n = 529, m = 212, bf16, 4/4 heads: a call 61 us with a thread per row, now 37)
// One head of 4 rows, n = 576, m = 231 in fp32: 39 -> 18 us between events (one load of theta in flight per thread and 64 rows of U at a time
// through shared memory before).
// RP: pitch of a position's 16 partial logits, 17 against bank conflicts, 16 where retained rows take the last of the shared memory
template <typename T, int RP>
__global__ void __launch_bounds__(256) expand_kernel(DecodeArgs a) {
  constexpr int R16 = EXP_ROWS;
  static_assert(EXP_ROWS == 16 && EXP_IC == 64, "thread mapping");
  extern __shared__ __align__(16) float smem[];
  const int ms = a.ms, m = a.m, n = a.n, msv = a.msv, mv = a.mv;
  float* Ssm = smem;                          // [ms][16]
  float* Wacc = Ssm + R16 * ms;               // [msv][16]
  float* red = Wacc + R16 * msv;              // [4][64][RP] partial logits of the quarters
  float* Psm = red + 4 * EXP_IC * RP;  // [64][16]
  float* rowmax = Psm + EXP_IC * R16;         // [16]
  float* rowsum = rowmax + R16;
  float* rowscale = rowsum + R16;

  const int split = blockIdx.x, rt = blockIdx.y, h = blockIdx.z;
  const int nrows_h = a.B * a.G * a.R;
  const int row0 = rt * R16;
  const int i_begin = split * a.ws.IR, i_end = min(n, i_begin + a.ws.IR);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const T* theta = static_cast<const T*>(a.theta) + (size_t)h * m * n;
  const T* U = static_cast<const T*>(a.U) + (size_t)h * mv * n;
  const float* S = a.S + (size_t)h * nrows_h * ms;
  const int ii = tid & 63, qd = tid >> 6;     // position in the chunk, quarter of the retained rows
  // 16-byte loads of U: rows start on 16-byte boundaries.  U read from L2 by its rows' threads: in bf16 only so and where there are enough of
  // them to keep the warps busy; in fp32 always (staged it was 24 % faster to 11 % slower over 60 calls of other block lengths)
  constexpr int EPV = Elems16<T>::N;
  const bool vec = n % EPV == 0 && (reinterpret_cast<uintptr_t>(U) & 15) == 0;
  const bool direct = sizeof(T) == sizeof(float) || (vec && mv > 64);

  grid_dep_wait();
  grid_dep_launch();
  for (int x = tid; x < R16 * ms; x += 256) {
    const int r = x / ms, j = x - r * ms;
    Ssm[j * R16 + r] = (row0 + r < nrows_h && j < m) ? S[(size_t)(row0 + r) * ms + j] : 0.f;
  }
  for (int x = tid; x < R16 * msv; x += 256) Wacc[x] = 0.f;
  if (tid < R16) { rowmax[tid] = -INFINITY; rowsum[tid] = 0.f; }
  __syncthreads();

  auto fma16 = [](float (&acc)[R16], const float* v, float x) {      // acc += v[0..15] x, v in shared memory
#pragma unroll
    for (int k = 0; k < R16; k += 4) {
      const float4 s = *reinterpret_cast<const float4*>(v + k);
      acc[k] = fmaf(s.x, x, acc[k]); acc[k + 1] = fmaf(s.y, x, acc[k + 1]);
      acc[k + 2] = fmaf(s.z, x, acc[k + 2]); acc[k + 3] = fmaf(s.w, x, acc[k + 3]);
    }
  };
  for (int i0 = i_begin; i0 < i_end; i0 += EXP_IC) {
    // ---- L chunk [16 rows x 64] = S theta[:, i0 : i0 + 64]
    const bool ok = i0 + ii < i_end;
    {
      float acc[R16];
#pragma unroll
      for (int k = 0; k < R16; ++k) acc[k] = 0.f;
      if (ok && a.id_theta) {
        if (qd == 0) fma16(acc, Ssm + (size_t)(i0 + ii) * R16, 1.f);
      } else if (ok) {
        const T* tp = theta + i0 + ii;
        int j = qd;
        for (; j + 28 < m; j += 32) {
          float t[8];
#pragma unroll
          for (int e = 0; e < 8; ++e) t[e] = to_f32(tp[(size_t)(j + 4 * e) * n]);
#pragma unroll
          for (int e = 0; e < 8; ++e) fma16(acc, Ssm + (size_t)(j + 4 * e) * R16, t[e]);
        }
        for (; j < m; j += 4) fma16(acc, Ssm + (size_t)j * R16, to_f32(tp[(size_t)j * n]));
      }
#pragma unroll
      for (int k = 0; k < R16; ++k) red[(qd * EXP_IC + ii) * RP + k] = acc[k];
    }
    __syncthreads();
    // ---- running max, P = exp(L - max), running sum: warp w owns rows 2w and 2w + 1
#pragma unroll
    for (int rr = 0; rr < 2; ++rr) {
      const int r = warp * 2 + rr;
      float l[2];
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        const int c = lane + 32 * x;
        float v = 0.f;
#pragma unroll
        for (int q = 0; q < 4; ++q) v += red[(q * EXP_IC + c) * RP + r];
        l[x] = i0 + c < i_end ? v : -INFINITY;
      }
      float cm = fmaxf(l[0], l[1]);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) cm = fmaxf(cm, __shfl_xor_sync(0xffffffffu, cm, o));
      const float m_old = rowmax[r], m_new = fmaxf(m_old, cm);
      const float p0 = __expf(l[0] - m_new), p1 = __expf(l[1] - m_new);
      float ps = p0 + p1;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) ps += __shfl_xor_sync(0xffffffffu, ps, o);
      Psm[lane * R16 + r] = p0;
      Psm[(lane + 32) * R16 + r] = p1;
      __syncwarp();
      if (lane == 0) {
        const float sc = (m_old == -INFINITY) ? 0.f : __expf(m_old - m_new);
        rowscale[r] = sc;
        rowsum[r] = rowsum[r] * sc + ps;
        rowmax[r] = m_new;
      }
    }
    __syncthreads();
    if (a.id_U) {
      // W = P: the columns of this CTA's range written so far follow the running maximum, the chunk's columns are P
      for (int x = tid; x < R16 * (i0 - i_begin); x += 256) Wacc[i_begin * R16 + x] *= rowscale[x & (R16 - 1)];
      for (int x = tid; x < R16 * min(EXP_IC, i_end - i0); x += 256) Wacc[i0 * R16 + x] = Psm[x];
      __syncthreads();
      continue;
    }
    // ---- W[:, j] = W[:, j] * scale + P . U[j, i0 : i0 + 64]^T
    const int cnt = min(EXP_IC, i_end - i0);
    if (direct) {
      for (int j = tid; j < mv; j += 256) {
        float acc[R16];
#pragma unroll
        for (int k = 0; k < R16; k += 4) {
          const float4 w = *reinterpret_cast<const float4*>(Wacc + (size_t)j * R16 + k), sc = *reinterpret_cast<const float4*>(rowscale + k);
          acc[k] = w.x * sc.x; acc[k + 1] = w.y * sc.y; acc[k + 2] = w.z * sc.z; acc[k + 3] = w.w * sc.w;
        }
        const T* up = U + (size_t)j * n + i0;
        int i = 0;
        for (; vec && i + 4 * EPV <= cnt; i += 4 * EPV) {
          float u[4][EPV];
#pragma unroll
          for (int v = 0; v < 4; ++v) load16(up + i + v * EPV, u[v]);
#pragma unroll
          for (int v = 0; v < 4; ++v)
#pragma unroll
            for (int e = 0; e < EPV; ++e) fma16(acc, Psm + (i + v * EPV + e) * R16, u[v][e]);
        }
        for (; i < cnt; ++i) fma16(acc, Psm + i * R16, to_f32(up[i]));
#pragma unroll
        for (int k = 0; k < R16; k += 4) *reinterpret_cast<float4*>(Wacc + (size_t)j * R16 + k) = make_float4(acc[k], acc[k + 1], acc[k + 2], acc[k + 3]);
      }
      __syncthreads();
    } else {
      // 64 rows of U at a time through shared memory (the partial logits' region), each row turned by its number against bank conflicts
      for (int j0 = 0; j0 < mv; j0 += 64) {
#pragma unroll
        for (int x = 0; x < 16; ++x) {
          const int jj = qd + 4 * x;
          red[jj * 64 + ((ii + jj) & 63)] = j0 + jj < mv && ii < cnt ? to_f32(U[(size_t)(j0 + jj) * n + i0 + ii]) : 0.f;
        }
        __syncthreads();
        if (j0 + ii < mv) {
          float4* wp = reinterpret_cast<float4*>(Wacc + (size_t)(j0 + ii) * R16 + qd * 4);
          const float4 w = *wp, sc = *reinterpret_cast<const float4*>(rowscale + qd * 4);
          float4 acc = make_float4(w.x * sc.x, w.y * sc.y, w.z * sc.z, w.w * sc.w);
#pragma unroll 8
          for (int i = 0; i < cnt; ++i) {
            const float u = red[ii * 64 + ((i + ii) & 63)];
            const float4 p = *reinterpret_cast<const float4*>(Psm + i * R16 + qd * 4);
            acc.x = fmaf(p.x, u, acc.x); acc.y = fmaf(p.y, u, acc.y); acc.z = fmaf(p.z, u, acc.z); acc.w = fmaf(p.w, u, acc.w);
          }
          *wp = acc;
        }
        __syncthreads();
      }
    }
  }

  float* Wout = a.W + ((size_t)split * a.H_kv + h) * nrows_h * msv;
  for (int x = tid; x < R16 * msv; x += 256) {
    const int r = x / msv, j = x - r * msv;
    if (row0 + r < nrows_h) Wout[(size_t)(row0 + r) * msv + j] = Wacc[j * R16 + r];
  }
  if (tid < R16 && row0 + tid < nrows_h)
    a.wstat[((size_t)split * a.H_kv + h) * nrows_h + row0 + tid] = make_float2(rowmax[tid], rowsum[tid]);
}

// rho = 0: theta = U = I, so L_img = S_comp and W = P.  One warp per row; writes the combined format.
__global__ void __launch_bounds__(256) passthrough_softmax_kernel(DecodeArgs a) {
  grid_dep_wait();
  grid_dep_launch();
  const int nrows = a.H_kv * a.B * a.G * a.R;
  const int row = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (row >= nrows) return;
  const float* s = a.S + (size_t)row * a.ms;
  float* w = a.Wcomb + (size_t)row * a.ms;
  float mx = -INFINITY;
  for (int j = lane; j < a.m; j += 32) mx = fmaxf(mx, s[j]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  float sum = 0.f;
  for (int j = lane; j < a.ms; j += 32) {
    const float p = j < a.m ? __expf(s[j] - mx) : 0.f;
    w[j] = p;
    sum += p;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if (lane == 0) a.statc[row] = make_float4(mx, sum, 0.f, 0.f);
}

// The n-split partials of one row combined relative to the row's overall maximum:
//   Wcomb[row][:] = sum_s e^{max_s - max} W_s[row][:],   statc[row] = (max, sum_s e^{max_s - max} sum_s).
// One warp per row (KV head, sequence, head in group, block).
__global__ void __launch_bounds__(256) combine_kernel(DecodeArgs a) {
  grid_dep_wait();
  grid_dep_launch();
  const int nrows = a.H_kv * a.B * a.G * a.R;
  const int row = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (row >= nrows) return;
  const int NS = a.ws.NS;
  float2 st = make_float2(-INFINITY, 0.f);
  if (lane < NS) st = a.wstat[(size_t)lane * nrows + row];
  float mx = st.x;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  const float my_sc = lane < NS ? __expf(st.x - mx) : 0.f;
  float sum = my_sc * st.y;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  float sc[MAX_NS];
#pragma unroll
  for (int s = 0; s < MAX_NS; ++s) sc[s] = __shfl_sync(0xffffffffu, my_sc, s);
  const size_t sstride = (size_t)nrows * a.msv;
  const float* wp = a.W + (size_t)row * a.msv;
  float* wo = a.Wcomb + (size_t)row * a.msv;
  for (int j = lane; j < a.msv; j += 32) {
    float v[MAX_NS];
#pragma unroll
    for (int s = 0; s < MAX_NS; ++s) v[s] = s < NS ? __ldcg(wp + s * sstride + j) : 0.f;
    float w = 0.f;
#pragma unroll
    for (int s = 0; s < MAX_NS; ++s) w = fmaf(sc[s], v[s], w);
    wo[j] = w;
  }
  if (lane == 0) a.statc[row] = make_float4(mx, sum, 0.f, 0.f);
}

static size_t expand_smem_bytes(int ms, int msv, int rp) {
  return sizeof(float) * ((size_t)EXP_ROWS * (ms + msv) + 4 * EXP_IC * rp + EXP_IC * EXP_ROWS + 3 * EXP_ROWS);
}

template <typename T, int RP>
static cudaError_t launch_expand_rp(const DecodeArgs& a, cudaStream_t st) {
  const size_t smem = expand_smem_bytes(a.ms, a.msv, RP);
  cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(expand_kernel<T, RP>), smem);
  if (e != cudaSuccess) return e;
  dim3 grid(a.ws.NS, ceil_div(a.B * a.G * a.R, EXP_ROWS), a.H_kv);
  // Programmatic overlap with the fp32 score kernel only (one sequence, one layer: 37.6 us per call, 40.7 without); behind the bf16 one, which
  // does not let it start early, it costs (32 sequences of one block of n = 81, 4/4 heads: 29.6 us per call, 21.7 without)
  if (sizeof(T) == sizeof(float)) return launch_dependent(expand_kernel<T, RP>, grid, dim3(256), smem, st, a);
  expand_kernel<T, RP><<<grid, 256, smem, st>>>(a);
  return cudaGetLastError();
}

template <typename T>
static cudaError_t launch_expand_t(const DecodeArgs& a, cudaStream_t st) {
  // 3280 and 3296 score and weight entries a row (rounded up to 16 each) are the most the two pitches leave room for
  return expand_smem_bytes(a.ms, a.msv, EXP_ROWS + 1) <= 227u * 1024u ? launch_expand_rp<T, EXP_ROWS + 1>(a, st) : launch_expand_rp<T, EXP_ROWS>(a, st);
}

cudaError_t launch_expand(const DecodeArgs& a, int dtype, cudaStream_t st) {
  if (a.R == 0) return cudaSuccess;
  const int nrows = a.H_kv * a.B * a.G * a.R;
  if (a.passthrough) {
    ProfScope prof(KVC_KERNEL_EXPAND, st);
    return launch_dependent(passthrough_softmax_kernel, dim3(ceil_div(nrows, 8)), dim3(256), 0, st, a);
  }
  cudaError_t e;
  {
    ProfScope prof(KVC_KERNEL_EXPAND, st);
    if (a.ws.use_mma) e = launch_expand_mma(a, st);
    else e = dtype == KVC_BF16 ? launch_expand_t<__nv_bfloat16>(a, st) : launch_expand_t<float>(a, st);
  }
  if (e != cudaSuccess) return e;
  ProfScope prof(KVC_KERNEL_COMBINE, st);
  return launch_dependent(combine_kernel, dim3(ceil_div(nrows, 8)), dim3(256), 0, st, a);
}

}  // namespace kvc
