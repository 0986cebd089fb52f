// Parameter fits from activations, on the device and in fp64 (calibration-time work, not the decode path):
//   FitValuePCA (App. C, Alg. 2; Sec. 3.1 "Sequence-Level Low-Rank Compression for Values"): mu = mean over the pooled
//     blocks and their n positions, U = the top m eigenvectors of the n x n token covariance of the centred values
//     (= the top m left singular vectors of the pooled centred columns);
//   the key reconstructor for a fixed retained index set as the minimiser of the reconstruction term of Alg. 2:
//     theta = (K_r K_r^T)^+ K_r K^T with K_r the retained rows, the pseudo-inverse taken through the eigen-decomposition.
// Both rest on a hand-written Jacobi solver for symmetric positive semidefinite matrices, in two forms:
//   up to 640 indices  one-sided (Hestenes): the columns of A + tau I are rotated in pairs until they are orthogonal; they then are
//                      sigma_i u_i with u_i the eigenvectors and sigma_i - tau the eigenvalues.  One launch, a cluster of CTAs per
//                      matrix (see jacobi_cluster_kernel)
//   beyond             two-sided cyclic with the round-robin ordering: the n/2 rotations of a round act on disjoint index pairs, so a
//                      round is one data-parallel update A <- J^T A J, Q <- Q J in which every 2 x 2 block of A is transformed in
//                      place by the rotations of its row pair and its column pair (two launches per round)
#include <vector>

#include "kvc_async.cuh"
#include "kvc_internal.cuh"

namespace kvc {

constexpr int FIT_TILE = 64;            // covariance tile per CTA
constexpr int FIT_KC = 32;              // channels per staged chunk
constexpr int FIT_SPLITS = 4;            // parts of the samples, one per matrix of the workspace
constexpr int FIT_MAX_SWEEPS = 40;
// one-sided: stop after a sweep whose largest squared cosine between two columns was below this.  Convergence is quadratic only between
// eigenvalues that stand apart: 32 blocks of n = 256 go 4e-7, 1e-12, 2e-26, but in a cluster, and fewer samples than positions always make one of
// the null space, the squares fall by a factor of ten a sweep (one block of 256: 8e-12, 8e-13, 7e-13, 3e-14, 3e-15, 2e-18, 8e-26), and a sweep
// may show a drop from elsewhere while the cluster's are still coming.  Stopped at 1e-11, rows of U were 1.2e-6 from orthonormal there, and
// eigenvalues equal to 1e-5 off by 1e-6 of the largest; 32 blocks of 256 took one sweep less, both fits 3.76 ms instead of 3.93
constexpr float FIT_COS_TOL2 = 1e-20f;
constexpr double FIT_OFF_TOL2 = 1e-22;  // stop when (off-diagonal norm / diagonal norm)^2 falls below this

static inline int even_up(int x) { return (x + 1) & ~1; }

// per-head regions of the fit workspace, in doubles
struct FitLayout {
  int ne;                 // n rounded up to even (the Jacobi pairing needs an even size; the extra index is all zero)
  size_t mat;             // ne * ne
  size_t off_M[4];        // four ne x ne matrices
  size_t off_lam;         // [ne]
  size_t off_inv;         // [ne]
  size_t off_rot;         // [ne] as double2 [ne / 2]
  size_t off_order;       // [ne] ints (in a region of ne doubles)
  size_t off_idx;         // [ne] ints
  size_t off_norm;        // [2]: off-diagonal and diagonal sums of squares
  size_t off_sum;         // [D]
  size_t off_flag;        // 64 floats: largest squared cosine of every sweep; an int at [60]: sweeps taken (one-sided solver)
  size_t per_head;
};

static FitLayout fit_layout(int n) {
  FitLayout f{};
  f.ne = even_up(n);
  f.mat = (size_t)f.ne * f.ne;
  size_t off = 0;
  for (int i = 0; i < 4; ++i) { f.off_M[i] = off; off += f.mat; }
  f.off_lam = off; off += f.ne;
  f.off_inv = off; off += f.ne;
  f.off_rot = off; off += f.ne;
  f.off_order = off; off += f.ne;
  f.off_idx = off; off += f.ne;
  f.off_norm = off; off += 2;
  f.off_sum = off; off += D;
  f.off_flag = off; off += 32;
  f.per_head = (off + 31) / 32 * 32;
  return f;
}

// ---- pooled sums and second moments ---------------------------------------------------------------------------
// sum[h][c] += sum over sequences and rows of X[b, h, row, c]
template <typename T>
__global__ void __launch_bounds__(256) fit_sum_kernel(const T* __restrict__ X, int B, int H_kv, long long rows, double* sum,
                                                      size_t head_stride) {
  const int h = blockIdx.x, c = threadIdx.x & (D - 1);
  const long long total = (long long)B * rows;
  double acc = 0.0;
  for (long long rr = (long long)blockIdx.y * 2 + (threadIdx.x >> 7); rr < total; rr += (long long)gridDim.y * 2) {
    const long long b = rr / rows, i = rr - b * rows;
    acc += (double)to_f32(X[((b * H_kv + h) * rows + i) * D + c]);
  }
  atomicAdd(sum + (size_t)h * head_stride + c, acc);
}

// Partial sums of the symmetric second-moment matrix: C_split[h][i][j] = sum over the split's blocks s and channels c of
// (X_s[i][c] - mu_c)(X_s[j][c] - mu_c), mu = sum / count (0 if !center).  Bound: fp64 multiply-adds (and as many shared-memory
// wavefronts).  Only tiles on and above the diagonal are computed, and the samples are split four ways into the four matrices of the
// workspace, so that a few heads fill the machine: n = 256, 32 samples, 4 heads 163 us (596 us for the full square in one piece, with
// each thread's columns side by side, which is a four-way bank conflict).
template <typename T>
__global__ void __launch_bounds__(256) fit_moment_kernel(const T* __restrict__ X, int B, int R, int H_kv, int n, int ne,
                                                         double* __restrict__ ws, size_t head_stride, size_t off_C, size_t mat,
                                                         size_t off_sum, int center) {
  __shared__ double As[FIT_KC][FIT_TILE], Bs[FIT_KC][FIT_TILE];
  __shared__ double mu[D];
  const int h = blockIdx.z, split = blockIdx.y;
  int ti = 0, tj = blockIdx.x;                              // tile (ti, tj), tj >= ti
  for (int row = (n + FIT_TILE - 1) / FIT_TILE; tj >= row; --row) { tj -= row; ++ti; }
  tj += ti;
  const int i0 = ti * FIT_TILE, j0 = tj * FIT_TILE;
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
  double* C = ws + (size_t)h * head_stride + off_C + (size_t)split * mat;
  const bool aligned = (reinterpret_cast<uintptr_t>(X) & 15) == 0;
  if (tid < D) mu[tid] = center ? ws[(size_t)h * head_stride + off_sum + tid] / ((double)B * R * n) : 0.0;
  __syncthreads();
  double acc[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[a][b] = 0.0;
  const int lrow = tid & 63, lc = (tid >> 6) * 8;          // staging: 64 rows x 4 groups of 8 channels, a warp along the rows
  const int s0 = (int)((long long)B * R * split / FIT_SPLITS), s1 = (int)((long long)B * R * (split + 1) / FIT_SPLITS);
  for (int s = s0; s < s1; ++s) {
    const int b = s / R, r = s - b * R;
    const T* blk = X + (((size_t)b * H_kv + h) * R + r) * (size_t)n * D;
    for (int c0 = 0; c0 < D; c0 += FIT_KC) {
#pragma unroll
      for (int side = 0; side < 2; ++side) {
        const int row = (side ? j0 : i0) + lrow;
        float f[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) f[e] = 0.f;
        if (row < n && !aligned) {
#pragma unroll
          for (int e = 0; e < 8; ++e) f[e] = to_f32(blk[(size_t)row * D + c0 + lc + e]);
        } else if (row < n) {
          constexpr int EPV = Elems16<T>::N;
#pragma unroll
          for (int v = 0; v < 8; v += EPV) {
            float x[EPV];
            load16(blk + (size_t)row * D + c0 + lc + v, x);
#pragma unroll
            for (int e = 0; e < EPV; ++e) f[v + e] = x[e];
          }
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) (side ? Bs : As)[lc + e][lrow] = row < n ? (double)f[e] - mu[c0 + lc + e] : 0.0;
      }
      __syncthreads();
#pragma unroll 8
      for (int k = 0; k < FIT_KC; ++k) {
        double av[4], bv[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) { av[e] = As[k][ty + 16 * e]; bv[e] = Bs[k][tx + 16 * e]; }
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int bb = 0; bb < 4; ++bb) acc[a][bb] = fma(av[a], bv[bb], acc[a][bb]);
      }
      __syncthreads();
    }
  }
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int bb = 0; bb < 4; ++bb) {
      const int i = i0 + ty + 16 * a, j = j0 + tx + 16 * bb;
      if (i < n && j < n) C[(size_t)i * ne + j] = acc[a][bb];
    }
}

// the splits summed into the first matrix, both triangles
__global__ void __launch_bounds__(256) fit_moment_sum_kernel(double* __restrict__ ws, size_t head_stride, size_t off_C, size_t mat, int n, int ne) {
  double* C = ws + (size_t)blockIdx.y * head_stride + off_C;
  for (int x = blockIdx.x * 256 + threadIdx.x; x < n * n; x += gridDim.x * 256) {
    const int i = x / n, j = x - i * n;
    if (j / FIT_TILE < i / FIT_TILE) continue;               // a tile below the diagonal: written by its mirror image
    double v = 0.0;
#pragma unroll
    for (int k = 0; k < FIT_SPLITS; ++k) v += C[(size_t)k * mat + (size_t)i * ne + j];
    C[(size_t)i * ne + j] = v;
    if (j / FIT_TILE > i / FIT_TILE) C[(size_t)j * ne + i] = v;
  }
}

// ---- cyclic Jacobi with the round-robin ordering --------------------------------------------------------------
// Round k of a sweep over an even number ne of indices: index ne-1 meets k; (k + j) mod (ne-1) meets (k - j) mod (ne-1).
__device__ __forceinline__ void round_pair(int k, int j, int ne, int& p, int& q) {
  const int nm1 = ne - 1;
  int a, b;
  if (j == 0) { a = nm1; b = k; }
  else { a = (k + j) % nm1; b = (k - j + nm1) % nm1; }
  p = a < b ? a : b;
  q = a < b ? b : a;
}

__global__ void jacobi_rotations_kernel(const double* __restrict__ ws, size_t head_stride, size_t off_A, size_t off_rot,
                                        int ne, int k, double* ws_out) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x, h = blockIdx.y;
  if (j >= ne / 2) return;
  const double* A = ws + (size_t)h * head_stride + off_A;
  int p, q;
  round_pair(k, j, ne, p, q);
  const double app = A[(size_t)p * ne + p], aqq = A[(size_t)q * ne + q], apq = A[(size_t)p * ne + q];
  double c = 1.0, s = 0.0;
  if (fabs(apq) > 1e-300 && fabs(apq) > 1e-18 * sqrt(fabs(app) * fabs(aqq))) {
    const double th = (aqq - app) / (2.0 * apq);
    const double t = (th >= 0.0 ? 1.0 : -1.0) / (fabs(th) + sqrt(th * th + 1.0));
    c = 1.0 / sqrt(t * t + 1.0);
    s = t * c;
  }
  double2* rot = reinterpret_cast<double2*>(ws_out + (size_t)h * head_stride + off_rot);
  rot[j] = make_double2(c, s);
}

// A <- J^T A J on the 2 x 2 block (row pair ja, column pair jb); Q <- Q J on rows (2 ja, 2 ja + 1), column pair jb
__global__ void __launch_bounds__(128) jacobi_apply_kernel(double* __restrict__ ws, size_t head_stride, size_t off_A,
                                                           size_t off_Q, size_t off_rot, int ne, int k) {
  const int jb = blockIdx.x * blockDim.x + threadIdx.x, ja = blockIdx.y, h = blockIdx.z;
  if (jb >= ne / 2) return;
  double* A = ws + (size_t)h * head_stride + off_A;
  double* Q = ws + (size_t)h * head_stride + off_Q;
  const double2* rot = reinterpret_cast<const double2*>(ws + (size_t)h * head_stride + off_rot);
  int p, q, pc, qc;
  round_pair(k, ja, ne, p, q);
  round_pair(k, jb, ne, pc, qc);
  const double2 ra = rot[ja], rb = rot[jb];
  const double b00 = A[(size_t)p * ne + pc], b01 = A[(size_t)p * ne + qc];
  const double b10 = A[(size_t)q * ne + pc], b11 = A[(size_t)q * ne + qc];
  // rows: J_a^T B
  const double x00 = ra.x * b00 - ra.y * b10, x01 = ra.x * b01 - ra.y * b11;
  const double x10 = ra.y * b00 + ra.x * b10, x11 = ra.y * b01 + ra.x * b11;
  // columns: (.) J_b
  double y00 = rb.x * x00 - rb.y * x01, y01 = rb.y * x00 + rb.x * x01;
  double y10 = rb.x * x10 - rb.y * x11, y11 = rb.y * x10 + rb.x * x11;
  if (ja == jb) { y01 = 0.0; y10 = 0.0; }                      // the annihilated pair, exactly
  A[(size_t)p * ne + pc] = y00; A[(size_t)p * ne + qc] = y01;
  A[(size_t)q * ne + pc] = y10; A[(size_t)q * ne + qc] = y11;
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    const size_t row = (size_t)(2 * ja + e) * ne;
    const double u = Q[row + pc], v = Q[row + qc];
    Q[row + pc] = rb.x * u - rb.y * v;
    Q[row + qc] = rb.y * u + rb.x * v;
  }
}

__global__ void __launch_bounds__(256) fit_norms_kernel(double* __restrict__ ws, size_t head_stride, size_t off_A,
                                                        size_t off_norm, int ne) {
  __shared__ double red[2][8];
  const int h = blockIdx.y;
  const double* A = ws + (size_t)h * head_stride + off_A;
  double off = 0.0, dg = 0.0;
  for (size_t x = (size_t)blockIdx.x * 256 + threadIdx.x; x < (size_t)ne * ne; x += (size_t)gridDim.x * 256) {
    const size_t i = x / ne, j = x - i * ne;
    const double v = A[x];
    if (i == j) dg += v * v; else off += v * v;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    off += __shfl_xor_sync(0xffffffffu, off, o);
    dg += __shfl_xor_sync(0xffffffffu, dg, o);
  }
  if ((threadIdx.x & 31) == 0) { red[0][threadIdx.x >> 5] = off; red[1][threadIdx.x >> 5] = dg; }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) { off += red[0][w]; dg += red[1][w]; }
    atomicAdd(ws + (size_t)h * head_stride + off_norm, off);
    atomicAdd(ws + (size_t)h * head_stride + off_norm + 1, dg);
  }
}

__global__ void fit_identity_kernel(double* __restrict__ ws, size_t head_stride, size_t off_Q, int ne) {
  const int h = blockIdx.y;
  double* Q = ws + (size_t)h * head_stride + off_Q;
  for (size_t x = (size_t)blockIdx.x * blockDim.x + threadIdx.x; x < (size_t)ne * ne; x += (size_t)gridDim.x * blockDim.x)
    Q[x] = (x / ne == x % ne) ? 1.0 : 0.0;
}

// eigenvalues = the diagonal; order[rank] = index, descending (ties by index; indices >= n_valid go last)
__global__ void fit_rank_kernel(double* __restrict__ ws, size_t head_stride, size_t off_A, size_t off_lam, size_t off_order,
                                int ne, int n_valid) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x, h = blockIdx.y;
  if (i >= ne) return;
  const double* A = ws + (size_t)h * head_stride + off_A;
  double* lam = ws + (size_t)h * head_stride + off_lam;
  int* order = reinterpret_cast<int*>(ws + (size_t)h * head_stride + off_order);
  const double li = A[(size_t)i * ne + i];
  int rank = 0;
  for (int j = 0; j < ne; ++j) {
    const double lj = A[(size_t)j * ne + j];
    const bool vi = i < n_valid, vj = j < n_valid;
    const bool before = (vj && !vi) || (vi == vj && (lj > li || (lj == li && j < i)));
    rank += before ? 1 : 0;
  }
  order[rank] = i;
  lam[i] = li;
}

// U[h][j][:] = eigenvector of rank j, sign fixed so that its entry of largest magnitude is positive
template <typename T>
__global__ void __launch_bounds__(128) fit_emit_basis_kernel(const double* __restrict__ ws, size_t head_stride, size_t off_Q,
                                                             size_t off_lam, size_t off_order, int ne, int n, int m,
                                                             T* __restrict__ U, double* __restrict__ eig) {
  __shared__ double best[4];
  __shared__ double sgn_s;
  const int j = blockIdx.x, h = blockIdx.y, tid = threadIdx.x;
  const double* Q = ws + (size_t)h * head_stride + off_Q;
  const int* order = reinterpret_cast<const int*>(ws + (size_t)h * head_stride + off_order);
  const int col = order[j];
  if (eig && tid == 0) eig[(size_t)h * n + j] = ws[(size_t)h * head_stride + off_lam + col];
  if (j >= m) return;
  double bv = 0.0;                       // entry of largest magnitude (first one on ties)
  for (int i = tid; i < n; i += 128) {
    const double v = Q[(size_t)i * ne + col];
    if (fabs(v) > fabs(bv)) bv = v;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double ov = __shfl_xor_sync(0xffffffffu, bv, o);
    if (fabs(ov) > fabs(bv)) bv = ov;
  }
  if ((tid & 31) == 0) best[tid >> 5] = bv;
  __syncthreads();
  if (tid == 0) {
    for (int w = 1; w < 4; ++w) if (fabs(best[w]) > fabs(bv)) bv = best[w];
    sgn_s = bv < 0.0 ? -1.0 : 1.0;
  }
  __syncthreads();
  const double sg = sgn_s;
  for (int i = tid; i < n; i += 128) store_elem(U + ((size_t)h * m + j) * n + i, (float)(sg * Q[(size_t)i * ne + col]));
}

template <typename T>
__global__ void fit_emit_mean_kernel(const double* __restrict__ ws, size_t head_stride, size_t off_sum, double count,
                                     T* __restrict__ mu) {
  const int h = blockIdx.x, c = threadIdx.x;
  store_elem(mu + h * D + c, (float)(ws[(size_t)h * head_stride + off_sum + c] / count));
}

// ---- least-squares pieces ------------------------------------------------------------------------------------
// A[j][j'] = C[idx[j]][idx[j']] (me x me, zero beyond m)
__global__ void fit_select_kernel(double* __restrict__ ws, size_t head_stride, size_t off_C, size_t off_A, size_t off_idx,
                                  int ne, int me, int m) {
  const int h = blockIdx.y;
  const double* C = ws + (size_t)h * head_stride + off_C;
  double* A = ws + (size_t)h * head_stride + off_A;
  const int* idx = reinterpret_cast<const int*>(ws + (size_t)h * head_stride + off_idx);
  for (size_t x = (size_t)blockIdx.x * blockDim.x + threadIdx.x; x < (size_t)me * me; x += (size_t)gridDim.x * blockDim.x) {
    const int j = (int)(x / me), k = (int)(x % me);
    A[x] = (j < m && k < m) ? C[(size_t)idx[j] * ne + idx[k]] : 0.0;
  }
}

// inv[i] = 1 / lam[i] where lam[i] > rcond * max lam, else 0 (one block per head)
__global__ void __launch_bounds__(256) fit_pinv_kernel(double* __restrict__ ws, size_t head_stride, size_t off_A, size_t off_inv,
                                                       int me, int m, double rcond) {
  __shared__ double red[8];
  const int h = blockIdx.x, tid = threadIdx.x;
  const double* A = ws + (size_t)h * head_stride + off_A;
  double mx = 0.0;
  for (int i = tid; i < me; i += 256) mx = fmax(mx, A[(size_t)i * me + i]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if ((tid & 31) == 0) red[tid >> 5] = mx;
  __syncthreads();
  mx = red[0];
  for (int w = 1; w < 8; ++w) mx = fmax(mx, red[w]);
  double* inv = ws + (size_t)h * head_stride + off_inv;
  for (int i = tid; i < me; i += 256) {
    const double l = A[(size_t)i * me + i];
    inv[i] = (l > 0.0 && l > rcond * mx) ? 1.0 / l : 0.0;
  }
  (void)m;
}

// T1[i][c] = inv[i] * sum_j Q[j][i] C[idx[j]][c]        (i < me, c < n)
__global__ void __launch_bounds__(256) fit_project_kernel(double* __restrict__ ws, size_t head_stride, size_t off_C, size_t off_Q,
                                                          size_t off_T, size_t off_inv, size_t off_idx, int ne, int me, int m,
                                                          int n) {
  __shared__ double Qs[16][17], Cs[16][17];
  const int h = blockIdx.z, i0 = blockIdx.y * 16, c0 = blockIdx.x * 16, ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
  const double* C = ws + (size_t)h * head_stride + off_C;
  const double* Q = ws + (size_t)h * head_stride + off_Q;
  const int* idx = reinterpret_cast<const int*>(ws + (size_t)h * head_stride + off_idx);
  double acc = 0.0;
  for (int j0 = 0; j0 < m; j0 += 16) {
    Qs[ty][tx] = (j0 + ty < m && i0 + tx < me) ? Q[(size_t)(j0 + ty) * me + i0 + tx] : 0.0;      // Qs[j][i]
    Cs[ty][tx] = (j0 + ty < m && c0 + tx < n) ? C[(size_t)idx[j0 + ty] * ne + c0 + tx] : 0.0;   // Cs[j][c]
    __syncthreads();
#pragma unroll
    for (int j = 0; j < 16; ++j) acc = fma(Qs[j][ty], Cs[j][tx], acc);
    __syncthreads();
  }
  if (i0 + ty < me && c0 + tx < n)
    ws[(size_t)h * head_stride + off_T + (size_t)(i0 + ty) * ne + c0 + tx] = acc * ws[(size_t)h * head_stride + off_inv + i0 + ty];
}

// theta[h][j][c] = sum_i Q[j][i] T1[i][c]
template <typename T>
__global__ void __launch_bounds__(256) fit_emit_theta_kernel(const double* __restrict__ ws, size_t head_stride, size_t off_Q,
                                                             size_t off_T, int ne, int me, int m, int n, T* __restrict__ theta) {
  __shared__ double Qs[16][17], Ts[16][17];
  const int h = blockIdx.z, j0 = blockIdx.y * 16, c0 = blockIdx.x * 16, ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
  const double* Q = ws + (size_t)h * head_stride + off_Q;
  const double* T1 = ws + (size_t)h * head_stride + off_T;
  double acc = 0.0;
  for (int i0 = 0; i0 < me; i0 += 16) {
    Qs[ty][tx] = (j0 + ty < m && i0 + tx < me) ? Q[(size_t)(j0 + ty) * me + i0 + tx] : 0.0;      // Qs[j][i]
    Ts[ty][tx] = (i0 + ty < me && c0 + tx < n) ? T1[(size_t)(i0 + ty) * ne + c0 + tx] : 0.0;    // Ts[i][c]
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 16; ++i) acc = fma(Qs[ty][i], Ts[i][tx], acc);
    __syncthreads();
  }
  if (j0 + ty < m && c0 + tx < n) store_elem(theta + ((size_t)h * m + j0 + ty) * n + c0 + tx, (float)acc);
}

// ---- one-sided Jacobi, one launch ----------------------------------------------------------------------------------------
// Bound: latency of a rotation (a dot product over a column reduced across a warp, the angle, the update; its warps issue in a quarter of the cycles), n - 1 of
// them one after the other per sweep whatever the machine's width, 12 to 15 sweeps, some 25 where there are fewer samples than positions.  So everything else is taken out of that chain: a
// cluster of C CTAs owns a matrix, its columns form 2 C blocks of bs, in each of the 2 C - 1 rounds of a sweep a CTA holds two blocks
// in shared memory (a warp per pair, the first block's column kept in registers) and rotates all pairs between them (in the first
// round also those inside), and between rounds the columns go to their next CTA behind one cluster barrier: through distributed shared
// memory up to 384 indices, beyond that (two buffers don't fit) through L2 (about 3 us per round); no launch, no host round trip.  Both
// fits of n = 256, m = 103, 4 heads on B200: 3.93 ms in 14 sweeps (at 13 sweeps 3.75, and 3.9 with the dot product reduced by shuffles, 4.3 also
// with the divisions and the square root of the angle rounded exactly and everything behind the dot product, 4.6 through L2; the two-sided
// form, two launches of 4 us per round, above 24).
// Half as many CTAs with twice the warps took a fifth longer (the rotations of 16 warps are bound by shared memory).
// The angle is taken in single precision, with approximate divisions: it only steers the convergence (off-diagonal cosines fall by 1e-7
// at worst per sweep once they are small); cosine and sine are made from its tangent in double precision, so that the rotation is
// orthogonal.  The squared lengths that the angle needs are carried along and taken anew in every round, and where one falls below a quarter; with them as two more dot products
// and the angle in double precision a rotation took 1.05 us where this took 0.89 then (both with their share of the rounds).
// tau = 1e-5 of the largest diagonal entry keeps the columns of a rank-deficient matrix away from zero, so that its null space gets
// orthonormal vectors too.
__device__ __forceinline__ float sqrt_approx(float x) {
  float y;
  asm("sqrt.approx.f32 %0, %1;\n" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ double ld_cluster_f64(uint32_t caddr) {
  double v;
  asm volatile("ld.shared::cluster.f64 %0, [%1];\n" : "=d"(v) : "r"(caddr) : "memory");
  return v;
}

// DS: the columns stay in shared memory, in two buffers (a round reads the peers' last one and writes the other); otherwise through L2
template <int EPL, bool DS>
__global__ void __launch_bounds__(640, 1) jacobi_cluster_kernel(double* __restrict__ ws, size_t head_stride, size_t off_A, size_t off_Q,
                                                                size_t off_flag, int size, int C, int bs) {
  constexpr int LD = 32 * EPL;
  extern __shared__ __align__(16) double cols_all[];             // [DS ? 2 : 1][2 bs][LD]
  double* cols = cols_all;
  __shared__ double s_red[32], s_norm[40];                       // s_norm: squared lengths of the block columns
  __shared__ float s_max[32];
  const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31, nw = bs;
  const int h = blockIdx.x / C, c = blockIdx.x - h * C, NB = 2 * C;
  double* A = ws + (size_t)h * head_stride + off_A;
  double* Q = ws + (size_t)h * head_stride + off_Q;
  float* flag = reinterpret_cast<float*>(ws + (size_t)h * head_stride + off_flag);
  double tau = 0.0;
  for (int i = tid; i < size; i += nw * 32) tau = fmax(tau, A[(size_t)i * size + i]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) tau = fmax(tau, __shfl_xor_sync(0xffffffffu, tau, o));
  if (lane == 0) s_red[w] = tau;
  __syncthreads();
  tau = 0.0;
  for (int x = 0; x < nw; ++x) tau = fmax(tau, s_red[x]);
  // the matrix is taken relative to its largest diagonal entry, so that the lengths are numbers of order one
  const double big = tau > 0.0 ? tau : 1.0, inv_big = 1.0 / big;
  tau = tau > 0.0 ? 1e-5 : 1.0;
  cluster_sync_all();                                            // every CTA has read the diagonal

  float mx = 0.f;
  auto length2 = [&](const double (&x)[EPL]) {
    double l = 0.0;
#pragma unroll
    for (int e = 0; e < EPL; ++e) l = fma(x[e], x[e], l);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
    return l;
  };
  // rotates columns a, b towards orthogonality; na, nb: their squared lengths, carried along
  auto rotate = [&](double (&a)[EPL], double (&b)[EPL], double& na, double& nb) {
    // what the angle needs of the lengths, made while the dot product is on its way (approximate: it only steers)
    // the lengths are numbers between 1e-10 and the size; 0 for an index beyond the matrix
    const float inv_len = rsqrtf((float)na) * rsqrtf((float)nb), half_diff = 0.5f * (float)(nb - na) * inv_len;
    const double scale = (double)inv_len * 0x1p30;
    double g0 = 0.0, g1 = 0.0;
#pragma unroll
    for (int e = 0; e < EPL; e += 2) { g0 = fma(a[e], b[e], g0); g1 = fma(a[e + 1], b[e + 1], g1); }
    const double g = g0 + g1;
    // the lanes' parts of the cosine in units of 2^-30 and the rests in units of 2^-56, as integers in the low words of sums with 1.5 * 2^52
    // (the parts together are at most the product of the lengths, 2^30, and 2^31 with lengths carried as below), so that two integer reductions
    // of the warp replace five steps of shuffles
    constexpr double MAGIC = 0x1.8p52;
    const double hi = fma(g, scale, MAGIC);
    const double lo = fma(fma(g, scale, MAGIC - hi), 0x1p26, MAGIC);
    const int hi_sum = __reduce_add_sync(0xffffffffu, __double2loint(hi)), lo_sum = __reduce_add_sync(0xffffffffu, __double2loint(lo));
    const float cosine = fmaf((float)lo_sum, 0x1p-56f, (float)hi_sum * 0x1p-30f);
    const float cos2 = cosine * cosine;
    if (!(cos2 > 1e-30f && inv_len > 0.f && inv_len < 1e30f)) return;
    mx = fmaxf(mx, cos2);
    // tangent of the angle: 1 / (z + sqrt(z^2 + 1)) with z = (nb - na) / (2 g), both sides times the cosine
    const float tf = __fdividef(half_diff >= 0.f ? cosine : -cosine, fabsf(half_diff) + sqrt_approx(fmaf(half_diff, half_diff, cos2)));
    const double ga = (double)__fdividef(cosine, inv_len);
    const double t = (double)tf, d = fma(t, t, 1.0);
    // 1 / sqrt(d): the approximation's relative error 1e-7 becomes its cube in one Halley step, and the rounding's
    double cs = (double)rsqrtf(fmaf(tf, tf, 1.f));
    const double err = fma(-d, cs * cs, 1.0);
    cs = fma(cs * err, fma(0.375, err, 0.5), cs);
    const double sn = cs * t;
    const double na0 = na, nb0 = nb;
    na = fma(-t, ga, na);
    nb = fma(t, ga, nb);
#pragma unroll
    for (int e = 0; e < EPL; ++e) {
      const double x = a[e], y = b[e];
      a[e] = cs * x - sn * y;
      b[e] = sn * x + cs * y;
    }
    // a column that was nearly parallel to the other loses most of its length, and what is left is no larger than the rounding of t ga: taken anew
    if (na < 0.25 * na0) na = length2(a);
    if (nb < 0.25 * nb0) nb = length2(b);
  };
  auto get = [&](double (&x)[EPL], int slot) {
#pragma unroll
    for (int e = 0; e < EPL; ++e) x[e] = cols[(size_t)slot * LD + e * 32 + lane];
  };
  auto put = [&](const double (&x)[EPL], int slot) {
#pragma unroll
    for (int e = 0; e < EPL; ++e) cols[(size_t)slot * LD + e * 32 + lane] = x[e];
  };
  auto fetch = [&](double (&x)[EPL], int col, bool shift) {
#pragma unroll
    for (int e = 0; e < EPL; ++e) {
      const int i = e * 32 + lane;
      x[e] = col < size && i < size ? __ldcg(A + (size_t)col * size + i) : 0.0;
      if (shift) x[e] *= inv_big;
      if (shift && i == col && col < size) x[e] += tau;
    }
  };
  auto save = [&](const double (&x)[EPL], int col) {
#pragma unroll
    for (int e = 0; e < EPL; ++e) {
      const int i = e * 32 + lane;
      if (col < size && i < size) __stcg(A + (size_t)col * size + i, x[e]);
    }
  };

  int sweep = 0;
  for (; sweep < FIT_MAX_SWEEPS;) {
    mx = 0.f;
    for (int br = 0; br < NB - 1; ++br) {
      // round robin over the blocks: block 0 stays, the others move one place per round; place c meets place NB - 1 - c
      auto at = [&](int pos) { return pos == 0 ? 0 : (pos - 1 - br + 2 * (NB - 1)) % (NB - 1) + 1; };
      const int p = at(c) * bs + w, q = at(NB - 1 - c) * bs + w;
      double a[EPL], b[EPL];
      const bool shift = sweep == 0 && br == 0;
      if (!DS || shift) {
        fetch(a, p, shift);
        fetch(b, q, shift);
      } else {
        // the block now in place x was in place x - 1 (the last for the first, block 0 stays), of CTA x or NB - 1 - x
        auto from = [&](int pos) {
          const int was = pos == 0 ? 0 : (pos == 1 ? NB - 1 : pos - 1);
          return map_to_cta(smem_addr(cols + (size_t)((was < C ? 0 : bs) + w) * LD + lane), (uint32_t)(was < C ? was : NB - 1 - was));
        };
        const uint32_t fa = from(c), fb = from(NB - 1 - c);
#pragma unroll
        for (int e = 0; e < EPL; ++e) { a[e] = ld_cluster_f64(fa + e * 256u); b[e] = ld_cluster_f64(fb + e * 256u); }
        cols = cols == cols_all ? cols_all + (size_t)2 * bs * LD : cols_all;
      }
      double na = length2(a), nb = length2(b);
      put(b, bs + w);
      if (lane == 0) s_norm[bs + w] = nb;
      if (br == 0) {
        put(a, w);
        if (lane == 0) s_norm[w] = na;
        __syncthreads();
        const int n2 = 2 * bs;
        for (int r = 0; r < n2 - 1; ++r) {
          auto place = [&](int pos) { return pos == 0 ? 0 : (pos - 1 - r + n2 - 1) % (n2 - 1) + 1; };
          const int i = place(w), j = place(n2 - 1 - w);
          get(a, i);
          get(b, j);
          na = s_norm[i];
          nb = s_norm[j];
          rotate(a, b, na, nb);
          put(a, i);
          put(b, j);
          __syncwarp();
          if (lane == 0) { s_norm[i] = na; s_norm[j] = nb; }
          __syncthreads();
        }
        get(a, w);
      } else {
        __syncthreads();
        int slot = bs + w;
        for (int r = 0; r < bs; ++r) {
          if (r > 0) { get(b, slot); nb = s_norm[slot]; }
          rotate(a, b, na, nb);
          put(b, slot);
          __syncwarp();
          if (lane == 0) s_norm[slot] = nb;
          slot = slot + 1 < 2 * bs ? slot + 1 : bs;
          __syncthreads();
        }
      }
      if (DS) {
        put(a, w);
      } else {
        save(a, p);
        get(b, bs + w);
        save(b, q);
      }
      if (br == NB - 2) {
        if (lane == 0) s_max[w] = mx;
        __syncthreads();
        if (tid == 0) {
          float m = 0.f;
          for (int x = 0; x < nw; ++x) m = fmaxf(m, s_max[x]);
          atomicMax(reinterpret_cast<int*>(flag) + sweep, __float_as_int(m));
        }
      }
      cluster_sync_all();                                        // the columns (and the sweep's maximum) can be read by their next owners
    }
    const float worst = __ldcg(flag + sweep);
    ++sweep;
    if (worst < FIT_COS_TOL2) break;
  }

  // the columns a warp finishes: the two it holds after the last round, or any two
  auto place_of = [&](int x) {
    if (!DS) return (2 * c + x) * bs + w;
    const int pos = x ? NB - 1 - c : c, br = NB - 2;
    return (pos == 0 ? 0 : (pos - 1 - br + 2 * (NB - 1)) % (NB - 1) + 1) * bs + w;
  };
  // eigenvalues and eigenvectors: Q[i][col] = column / its length, A[col][col] = length - tau
  double len[2];
#pragma unroll
  for (int x = 0; x < 2; ++x) {
    const int col = place_of(x);
    double a[EPL];
    if (DS) get(a, x * bs + w); else fetch(a, col, false);
    const double al = length2(a);
    len[x] = sqrt(al);
    const double inv = al > 0.0 ? 1.0 / len[x] : 0.0;
#pragma unroll
    for (int e = 0; e < EPL; ++e) {
      const int i = e * 32 + lane;
      if (col < size && i < size) Q[(size_t)i * size + col] = a[e] * inv;
    }
  }
  cluster_sync_all();                                            // every column has been read
#pragma unroll
  for (int x = 0; x < 2; ++x) {
    const int col = place_of(x);
    if (lane == 0 && col < size) A[(size_t)col * size + col] = (len[x] - tau) * (tau < 1.0 ? big : 0.0);
  }
  if (c == 0 && tid == 0) reinterpret_cast<int*>(flag)[60] = sweep;
}

// CTAs of a cluster: blocks of about eight columns, as many CTAs as the device places together (sixteen with the non-portable size)
template <int EPL>
static cudaError_t launch_jacobi_cluster(double* ws, size_t head_stride, size_t off_A, size_t off_Q, size_t off_flag, int H, int size,
                                         cudaStream_t st, bool* used) {
  constexpr bool DS = EPL <= 12;               // two buffers of columns fit shared memory up to 384 indices
  const void* fn = reinterpret_cast<const void*>(jacobi_cluster_kernel<EPL, DS>);
  *used = false;
  int C = ceil_div(size, 16);
  C = C > 16 ? 16 : C;
  const int bs = ceil_div(size, 2 * C);
  if (bs > 20) return cudaSuccess;
  const size_t smem = sizeof(double) * (DS ? 4 : 2) * (size_t)bs * 32 * EPL;
  cudaError_t e = ensure_dynamic_smem(fn, smem);
  if (e != cudaSuccess) return e;
  if (C > 8) e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(C * H));
  cfg.blockDim = dim3((unsigned)(bs * 32));
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)C; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int fit = 0;
  if (C > 8 && (cudaOccupancyMaxActiveClusters(&fit, fn, &cfg) != cudaSuccess || fit < 1)) { cudaGetLastError(); return cudaSuccess; }
  *used = true;
  return cudaLaunchKernelEx(&cfg, jacobi_cluster_kernel<EPL, DS>, ws, head_stride, off_A, off_Q, off_flag, size, C, bs);
}

// ---- host side -------------------------------------------------------------------------------------------------
// eigen-decomposition of the size x size matrices at off_A (overwritten by their diagonal form), eigenvectors to off_Q
// sweeps: one entry per head, complete when the stream has been synchronised
static cudaError_t jacobi_eigen(double* ws, const FitLayout& f, size_t off_A, size_t off_Q, int H, int size, cudaStream_t st,
                                std::vector<int>& sweeps) {
  const size_t head_stride = f.per_head, off_rot = f.off_rot, off_norm = f.off_norm;
  sweeps.assign(H, 0);
  {
    bool used = false;
    cudaError_t e = cudaSuccess;
#define KVC_JACOBI(EPL) launch_jacobi_cluster<EPL>(ws, head_stride, off_A, off_Q, f.off_flag, H, size, st, &used)
    if (size <= 64) e = KVC_JACOBI(2);
    else if (size <= 128) e = KVC_JACOBI(4);
    else if (size <= 256) e = KVC_JACOBI(8);
    else if (size <= 384) e = KVC_JACOBI(12);
    else if (size <= 640) e = KVC_JACOBI(20);
#undef KVC_JACOBI
    if (e != cudaSuccess) return e;
    if (used)
      return cudaMemcpy2DAsync(sweeps.data(), sizeof(int), reinterpret_cast<const int*>(ws + f.off_flag) + 60, head_stride * sizeof(double),
                               sizeof(int), (size_t)H, cudaMemcpyDeviceToHost, st);
  }
  fit_identity_kernel<<<dim3(64, H), 256, 0, st>>>(ws, head_stride, off_Q, size);
  cudaError_t e = cudaGetLastError();
  std::vector<double> norms((size_t)2 * H);
  int sweep = 0;
  for (; e == cudaSuccess && sweep < FIT_MAX_SWEEPS; ++sweep) {
    for (int h = 0; h < H && e == cudaSuccess; ++h)
      e = cudaMemsetAsync(ws + (size_t)h * head_stride + off_norm, 0, 2 * sizeof(double), st);
    if (e != cudaSuccess) break;
    fit_norms_kernel<<<dim3(32, H), 256, 0, st>>>(ws, head_stride, off_A, off_norm, size);
    for (int h = 0; h < H && e == cudaSuccess; ++h)
      e = cudaMemcpyAsync(&norms[2 * h], ws + (size_t)h * head_stride + off_norm, 2 * sizeof(double), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) break;
    bool done = true;
    for (int h = 0; h < H; ++h) done = done && !(norms[2 * h] > FIT_OFF_TOL2 * norms[2 * h + 1]);
    if (done) break;
    for (int k = 0; k < size - 1; ++k) {
      jacobi_rotations_kernel<<<dim3(ceil_div(size / 2, 128), H), 128, 0, st>>>(ws, head_stride, off_A, off_rot, size, k, ws);
      jacobi_apply_kernel<<<dim3(ceil_div(size / 2, 128), size / 2, H), 128, 0, st>>>(ws, head_stride, off_A, off_Q, off_rot, size, k);
    }
    e = cudaGetLastError();
  }
  sweeps.assign(H, sweep);
  return e;
}

// completes a fit: the stream is idle, the sweeps are known
static cudaError_t finish(cudaStream_t st, const std::vector<int>& sweeps, int* sweeps_out) {
  const cudaError_t e = cudaStreamSynchronize(st);
  if (e == cudaSuccess && sweeps_out) {
    *sweeps_out = 0;
    for (int s : sweeps) *sweeps_out = s > *sweeps_out ? s : *sweeps_out;
  }
  return e;
}

template <typename T>
static cudaError_t moments(const T* X, int B, int R, int H, int n, const FitLayout& f, double* ws, size_t off_C, bool center,
                           cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(ws, 0, (size_t)H * f.per_head * sizeof(double), st);
  if (e != cudaSuccess) return e;
  if (center) fit_sum_kernel<T><<<dim3(H, 64), 256, 0, st>>>(X, B, H, (long long)R * n, ws + f.off_sum, f.per_head);
  const int tiles = ceil_div(n, FIT_TILE);
  fit_moment_kernel<T><<<dim3(tiles * (tiles + 1) / 2, FIT_SPLITS, H), 256, 0, st>>>(X, B, R, H, n, f.ne, ws, f.per_head, off_C, f.mat, f.off_sum,
                                                                                   center ? 1 : 0);
  fit_moment_sum_kernel<<<dim3(ceil_div(n * n, 1024), H), 256, 0, st>>>(ws, f.per_head, off_C, f.mat, n, f.ne);
  return cudaGetLastError();
}

template <typename T>
static cudaError_t fit_pca_t(const void* V_vis, int B, int R, int H, int n, int m, void* U_out, void* mu_out, double* eig_out,
                             double* ws, cudaStream_t st, int* sweeps) {
  const FitLayout f = fit_layout(n);
  cudaError_t e = moments<T>(static_cast<const T*>(V_vis), B, R, H, n, f, ws, f.off_M[0], true, st);
  if (e != cudaSuccess) return e;
  std::vector<int> taken;
  e = jacobi_eigen(ws, f, f.off_M[0], f.off_M[1], H, f.ne, st, taken);
  if (e != cudaSuccess) return e;
  fit_rank_kernel<<<dim3(ceil_div(f.ne, 128), H), 128, 0, st>>>(ws, f.per_head, f.off_M[0], f.off_lam, f.off_order, f.ne, n);
  fit_emit_basis_kernel<T><<<dim3(eig_out ? n : m, H), 128, 0, st>>>(ws, f.per_head, f.off_M[1], f.off_lam, f.off_order, f.ne, n, m,
                                                                     static_cast<T*>(U_out), eig_out);
  fit_emit_mean_kernel<T><<<H, D, 0, st>>>(ws, f.per_head, f.off_sum, (double)B * R * n, static_cast<T*>(mu_out));
  e = cudaGetLastError();
  return e != cudaSuccess ? e : finish(st, taken, sweeps);
}

template <typename T>
static cudaError_t fit_theta_t(const void* K_vis, int B, int R, int H, int n, int m, const int32_t* idx, int idx_per_head,
                               double rcond, void* theta_out, double* ws, cudaStream_t st, int* sweeps) {
  const FitLayout f = fit_layout(n);
  const int me = even_up(m);
  cudaError_t e = moments<T>(static_cast<const T*>(K_vis), B, R, H, n, f, ws, f.off_M[0], false, st);
  for (int h = 0; h < H && e == cudaSuccess; ++h)
    e = cudaMemcpyAsync(ws + (size_t)h * f.per_head + f.off_idx, idx + (idx_per_head ? (size_t)h * m : 0), (size_t)m * sizeof(int32_t),
                        cudaMemcpyHostToDevice, st);
  if (e != cudaSuccess) return e;
  fit_select_kernel<<<dim3(64, H), 256, 0, st>>>(ws, f.per_head, f.off_M[0], f.off_M[1], f.off_idx, f.ne, me, m);
  std::vector<int> taken;
  e = jacobi_eigen(ws, f, f.off_M[1], f.off_M[2], H, me, st, taken);
  if (e != cudaSuccess) return e;
  fit_pinv_kernel<<<H, 256, 0, st>>>(ws, f.per_head, f.off_M[1], f.off_inv, me, m, rcond);
  fit_project_kernel<<<dim3(ceil_div(n, 16), ceil_div(me, 16), H), 256, 0, st>>>(ws, f.per_head, f.off_M[0], f.off_M[2], f.off_M[3],
                                                                              f.off_inv, f.off_idx, f.ne, me, m, n);
  fit_emit_theta_kernel<T><<<dim3(ceil_div(n, 16), ceil_div(m, 16), H), 256, 0, st>>>(ws, f.per_head, f.off_M[2], f.off_M[3], f.ne, me, m,
                                                                                    n, static_cast<T*>(theta_out));
  e = cudaGetLastError();
  return e != cudaSuccess ? e : finish(st, taken, sweeps);
}

}  // namespace kvc

using namespace kvc;

extern "C" {

size_t kvc_fit_workspace_bytes(int H_kv, int n) {
  if (H_kv < 1 || n < 1) return 0;
  return align_up((size_t)H_kv * fit_layout(n).per_head * sizeof(double), 256);
}

static int fit_args_ok(const void* X, int B, int R, int H_kv, int n, int m, int dtype, const void* out, const void* ws) {
  if (!X || !out || !ws) return KVC_ERR_ARG;
  if (B < 1 || R < 1 || H_kv < 1 || n < 1 || m < 1 || m > n || H_kv > 65535) return KVC_ERR_SHAPE;
  if (dtype != KVC_F32 && dtype != KVC_BF16) return KVC_ERR_DTYPE;
  if (reinterpret_cast<uintptr_t>(ws) & 255) return KVC_ERR_WORKSPACE;
  return KVC_OK;
}

int kvc_fit_value_pca(const void* V_vis, int B, int R, int H_kv, int n, int m, kvc_dtype dtype, void* U_out, void* mu_out,
                      double* eig_out, void* workspace, void* stream, int* sweeps_out) {
  const int s = fit_args_ok(V_vis, B, R, H_kv, n, m, (int)dtype, U_out, workspace);
  if (s != KVC_OK) return s;
  if (!mu_out) return KVC_ERR_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  double* ws = static_cast<double*>(workspace);
  return cuda_status(dtype == KVC_BF16
                         ? fit_pca_t<__nv_bfloat16>(V_vis, B, R, H_kv, n, m, U_out, mu_out, eig_out, ws, st, sweeps_out)
                         : fit_pca_t<float>(V_vis, B, R, H_kv, n, m, U_out, mu_out, eig_out, ws, st, sweeps_out));
}

int kvc_fit_key_reconstructor(const void* K_vis, int B, int R, int H_kv, int n, int m, const int32_t* idx, int idx_per_head,
                              double rcond, kvc_dtype dtype, void* theta_out, void* workspace, void* stream, int* sweeps_out) {
  const int s = fit_args_ok(K_vis, B, R, H_kv, n, m, (int)dtype, theta_out, workspace);
  if (s != KVC_OK) return s;
  if (!idx || !(rcond >= 0.0)) return KVC_ERR_ARG;
  for (int h = 0; h < (idx_per_head ? H_kv : 1); ++h)
    for (int j = 0; j < m; ++j) {
      const int32_t v = idx[(size_t)h * m + j];
      if (v < 0 || v >= n || (j > 0 && v <= idx[(size_t)h * m + j - 1])) return KVC_ERR_BOUNDS;
    }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  double* ws = static_cast<double*>(workspace);
  return cuda_status(dtype == KVC_BF16
                         ? fit_theta_t<__nv_bfloat16>(K_vis, B, R, H_kv, n, m, idx, idx_per_head, rcond, theta_out, ws, st, sweeps_out)
                         : fit_theta_t<float>(K_vis, B, R, H_kv, n, m, idx, idx_per_head, rcond, theta_out, ws, st, sweeps_out));
}

}  // extern "C"
