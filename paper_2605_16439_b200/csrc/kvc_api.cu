// Host side of the C ABI: validation, layer handles, workspace layout, kernel sequencing.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <map>
#include <mutex>
#include <new>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "kvc_internal.cuh"
#include "kvc_split.cuh"
#include "kvc_resident.cuh"
#include "kvc_cluster.cuh"
#include "kvc_plain.cuh"
#include "kvc_spread.cuh"

namespace kvc {

static size_t elem_bytes(int dtype) { return dtype == KVC_BF16 ? 2 : 4; }

WsLayout ws_layout(const kvc_layer* L, int B, int R, int T_cap, int forms) {
  WsLayout w{};
  const int H_kv = L->desc.H_kv, G = L->G, n = L->desc.n;
  const int ms = (L->mk + 15) / 16 * 16, msv = (L->mv + 15) / 16 * 16;
  const int rows_h = B * G * R;
  // tensor-core expansion: bf16 storage and 16-byte aligned rows of theta / U
  w.use_mma = (!L->passthrough && L->mode == KVC_MODE_KV && L->desc.dtype == KVC_BF16 && n % 8 == 0) ? 1 : 0;
  w.CG = 1;
  w.cgw = ms;
  int row_tiles;
  if (w.use_mma) {
    w.CG = ceil_div(ms, 256);
    w.cgw = (int)align_up((size_t)ceil_div(ms, w.CG), 16);
    // the kernel keeps a 64-row score tile and a chunk of theta over all retained positions in shared memory: past about 720
    // of them (n = 1024 at ratios below 0.3) that no longer fits, and the fp32 expansion takes over
    if (expand_mma_smem_bytes(ms, w.cgw) > 227u * 1024u) { w.use_mma = 0; w.CG = 1; w.cgw = ms; }
  }
  if (w.use_mma) {
    row_tiles = ceil_div(rows_h, 64) * H_kv * w.CG;
  } else {
    row_tiles = ceil_div(rows_h, EXP_ROWS) * H_kv;
  }
  if (L->passthrough || rows_h == 0) {
    w.NS = 1;
    w.IR = (int)align_up(n, EXP_IC);
  } else {
    int ns = ceil_div(EXP_TARGET_CTAS, row_tiles);
    ns = ns < 1 ? 1 : ns;
    int max_ns = ceil_div(n, EXP_IC);
    max_ns = max_ns > MAX_NS ? MAX_NS : max_ns;
    ns = ns > max_ns ? max_ns : ns;
    w.IR = (int)align_up((size_t)ceil_div(n, ns), EXP_IC);
    w.NS = ceil_div(n, w.IR);
  }
  w.cpb = ceil_div(L->mv, OUT_CHUNK);
  w.ct = ceil_div(T_cap, OUT_CHUNK);
  w.chunks_per_bh = R * w.cpb + w.ct;
  w.GT = G == 1 ? 1 : (G == 2 ? 2 : (G <= 4 ? 4 : 8));
  {
    const long long total = (long long)B * H_kv * w.chunks_per_bh;
    const int per_sm = w.GT <= 2 ? 3 : 2;
    long long ctas = (long long)(L->num_sms > 0 ? L->num_sms : 148) * per_sm;
    if (ctas > total) ctas = total;
    if (ctas < 1) ctas = 1;
    w.cpc = (int)((total + ctas - 1) / ctas);
    if (w.cpc < 1) w.cpc = 1;
    w.out_ctas = (int)((total + w.cpc - 1) / w.cpc);
  }
  {
    // a (sequence, KV head) spans chunks_per_bh <= cpc * ctas / (B*H_kv) chunks, hence at most that many + 1 CTAs;
    // the bound does not depend on T, so a workspace sized for T_cap fits every T <= T_cap
    const long long ctas_max = (long long)(L->num_sms > 0 ? L->num_sms : 148) * (w.GT <= 2 ? 3 : 2);
    const long long bh = (long long)B * H_kv;
    w.nsplit = (int)((ctas_max + (bh > 0 ? bh : 1) - 1) / (bh > 0 ? bh : 1)) + 2;
  }
  w.Ts = (int)align_up((size_t)(T_cap > 0 ? T_cap : 1), 4);
  size_t off = 0;
  auto take = [&](size_t bytes) { size_t o = off; off = align_up(off + bytes, 256); return o; };
  w.off_cnt = take(sizeof(int) * ((size_t)B * H_kv + 1));
  w.off_S = take((w.use_mma ? sizeof(__nv_bfloat16) : sizeof(float)) * (size_t)H_kv * rows_h * ms);
  w.off_stxt = take(sizeof(float) * (size_t)B * H_kv * G * w.Ts);
  w.off_W = take(sizeof(float) * (size_t)w.NS * H_kv * rows_h * msv);
  w.off_wstat = take(sizeof(float2) * (size_t)w.NS * H_kv * rows_h);
  w.off_Wc = take(sizeof(float) * (size_t)H_kv * rows_h * msv);
  w.off_statc = take(sizeof(float4) * (size_t)H_kv * rows_h);
  w.off_ypart = take(sizeof(float) * (size_t)B * H_kv * G * w.nsplit * D);
  w.off_ystat = take(sizeof(float2) * (size_t)B * H_kv * G * w.nsplit);
  {
    // partial outputs of the one-kernel path: per (sequence, KV head) one per unit along the block axis
    size_t np = 0;
    if (B > 0 && R > 0) {
      for (int ragged = 0; ragged < 2; ++ragged) {
        if (!(forms & (ragged ? WS_RAGGED : WS_UNIFORM))) continue;
        const FusedPlan fp = plan_fused(L, B, R, ragged != 0);
        if (fp.ok && L->mode == KVC_MODE_KV && fp.nrg > 1) np = std::max(np, (size_t)B * H_kv * fp.nrg * G);
      }
    }
    w.off_fpy = take(sizeof(float) * np * D);
    w.off_fpml = take(sizeof(float2) * np);
    w.off_fcnt = take(sizeof(unsigned long long) * (np ? (size_t)B * H_kv : 0));
  }
  {
    size_t sb = 0;
    if (B > 0 && R > 0) {
      const SplitPlan sp = plan_split(L, B, R);
      if (sp.ok && L->mode == KVC_MODE_KV) sb = split_ws(L, sp, B, R, T_cap).bytes;
    }
    w.off_split = take(sb);
  }
  w.off_resident = take(B > 0 && R > 0 && plan_resident(L, B, R, 0).ok ? resident_ws(L, B).bytes : 0);
  w.total = off;
  return w;
}

}  // namespace kvc

using namespace kvc;

namespace kvc {
cudaError_t ensure_dynamic_smem(const void* kernel, size_t bytes) {
  static std::mutex mu;
  static std::map<std::pair<const void*, int>, size_t> set_to;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lock(mu);
  size_t& have = set_to[std::make_pair(kernel, dev)];
  if (have >= bytes) return cudaSuccess;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e == cudaSuccess) have = bytes;
  return e;
}

static thread_local cudaError_t g_last_cuda = cudaSuccess;
// KVC_OK, or KVC_ERR_CUDA after remembering the error for kvc_last_cuda_error (the runtime's own slot is cleared)
int cuda_status(cudaError_t e) {
  if (e == cudaSuccess) return KVC_OK;
  g_last_cuda = e;
  cudaGetLastError();
  return KVC_ERR_CUDA;
}
}  // namespace kvc

extern "C" {

const char* kvc_last_cuda_error(void) { return cudaGetErrorString(g_last_cuda); }

int kvc_retained_len(int n, int ratio_permille) {
  if (n <= 0 || ratio_permille < 0 || ratio_permille >= 1000) return -1;
  return (int)(((long long)n * (1000 - ratio_permille) + 999) / 1000);
}

const char* kvc_strerror(int s) {
  switch (s) {
    case KVC_OK: return "ok";
    case KVC_ERR_ARG: return "invalid argument (null pointer or negative size)";
    case KVC_ERR_SHAPE: return "unsupported or inconsistent shape";
    case KVC_ERR_DTYPE: return "unknown dtype";
    case KVC_ERR_NO_PARAMS: return "theta / U / mu / idx missing for a compression ratio > 0";
    case KVC_ERR_WORKSPACE: return "workspace null, not 256-byte aligned, or static scratch too small for this shape";
    case KVC_ERR_CUDA: return "CUDA runtime error";
    case KVC_ERR_TIMEOUT: return "bounded device-side wait gave up";
    case KVC_ERR_BOUNDS: return "index set entry out of range or not strictly increasing";
    default: return "unknown status";
  }
}

int kvc_layer_create(const kvc_layer_desc* desc, kvc_layer** out) {
  if (!desc || !out) return KVC_ERR_ARG;
  *out = nullptr;
  if (desc->dtype != KVC_F32 && desc->dtype != KVC_BF16) return KVC_ERR_DTYPE;
  if (desc->d != D || desc->H_q <= 0 || desc->H_kv <= 0 || desc->H_q % desc->H_kv != 0 ||
      desc->H_q / desc->H_kv > MAX_G || desc->n <= 0)
    return KVC_ERR_SHAPE;
  const int m = kvc_retained_len(desc->n, desc->ratio_permille);
  if (m < 1) return KVC_ERR_SHAPE;
  const bool pass = desc->ratio_permille == 0;
  const int mode = pass ? KVC_MODE_KV : desc->mode;
  if (mode != KVC_MODE_KV && mode != KVC_MODE_K_ONLY && mode != KVC_MODE_V_ONLY) return KVC_ERR_ARG;
  const bool key_side = mode != KVC_MODE_V_ONLY, value_side = mode != KVC_MODE_K_ONLY;   // sides that are compressed
  if (!pass && ((key_side && (!desc->idx || !desc->theta)) || (value_side && (!desc->U || !desc->mu)))) return KVC_ERR_NO_PARAMS;

  std::vector<int32_t> idx((size_t)desc->H_kv * m);
  for (int h = 0; h < desc->H_kv; ++h)
    for (int j = 0; j < m; ++j) {
      const int32_t v = (pass || !key_side) ? j : desc->idx[(desc->idx_per_head ? (size_t)h * m : 0) + j];
      if (v < 0 || v >= desc->n || (j > 0 && v <= idx[(size_t)h * m + j - 1])) return KVC_ERR_BOUNDS;
      idx[(size_t)h * m + j] = v;
    }

  kvc_layer* L = new (std::nothrow) kvc_layer();
  if (!L) return KVC_ERR_ARG;
  L->desc = *desc;
  L->desc.idx = nullptr;
  L->m = m;
  L->ms = (m + 15) / 16 * 16;
  L->G = desc->H_q / desc->H_kv;
  L->passthrough = pass ? 1 : 0;
  L->capsules_fresh = 1;
  L->mode = mode;
  L->mk = key_side ? m : desc->n;
  L->mv = value_side ? m : desc->n;
  L->d_block = nullptr;
  L->d_idx = nullptr;
  L->d_cstatus = nullptr;
  L->d_usum = nullptr;
  L->maps = map_cache_create();
  L->num_sms = 0;
  std::memset(L->clusters, 0, sizeof(L->clusters));
  {
    const char* ex = std::getenv("KVC_EXPANSION");
    L->use_tc = !ex ? 0 : (std::strcmp(ex, "tcgen05") == 0 ? 1 : (std::strcmp(ex, "pair") == 0 ? 2 : (std::strcmp(ex, "mma") == 0 ? -1 : (std::strcmp(ex, "phases") == 0 ? -2 : (std::strcmp(ex, "split") == 0 ? 3 : (std::strcmp(ex, "resident") == 0 ? 4 : (std::strcmp(ex, "cluster") == 0 ? 5 : (std::strcmp(ex, "spread") == 0 ? 6 : 0))))))));
  }
  // one allocation: index set, status word, row sums of U, and where a kernel would read them, copies of theta and U with rows the TMA
  // engine can address (bf16): theta for the cluster path, whose tensor map cuts rows in groups of 64, U where its rows do not start on 16 bytes
  const int np = (int)align_up((size_t)desc->n, 64);
  const bool pad_theta = np != desc->n && (cluster_may_serve(L) || (spread_may_serve(L) && desc->n % 8 != 0));
  const bool pad_U = desc->dtype == KVC_BF16 && !pass && value_side && np != desc->n &&
                     (desc->n % 8 != 0 || !tma_rows(desc->U));
  L->theta_np = pad_theta ? np : desc->n;
  L->U_np = pad_U ? np : desc->n;
  L->theta_rows = key_side && !pass && np == desc->n ? desc->theta : nullptr;
  L->U_rows = value_side && !pass ? desc->U : nullptr;
  const size_t rows = (size_t)desc->H_kv * m, padded = rows * np * sizeof(__nv_bfloat16);
  size_t bytes = 0;
  auto take = [&](size_t b) { const size_t o = bytes; bytes = align_up(bytes + b, 256); return o; };
  const size_t o_idx = take(rows * sizeof(int32_t)), o_status = take(sizeof(int));
  const size_t o_usum = take(!pass && value_side ? rows * sizeof(float) : 0);
  const size_t o_theta = take(pad_theta ? padded : 0), o_U = take(pad_U ? padded : 0);
  cudaError_t e = cudaGetDevice(&L->device);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&L->num_sms, cudaDevAttrMultiProcessorCount, L->device);
  if (e == cudaSuccess && (cluster_may_serve(L) || spread_may_serve(L) || spread_f32_may_serve(L))) cluster_occupancy(L->device, L->num_sms, L->clusters);
  if (e == cudaSuccess) e = cudaMalloc(&L->d_block, bytes);
  if (e == cudaSuccess) {
    char* base = static_cast<char*>(L->d_block);
    L->d_idx = reinterpret_cast<int32_t*>(base + o_idx);
    L->d_cstatus = reinterpret_cast<int*>(base + o_status);
    e = cudaMemcpy(L->d_idx, idx.data(), idx.size() * sizeof(int32_t), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(L->d_cstatus, 0, sizeof(int));
    // theta and U may still be on their way on any stream
    if (e == cudaSuccess && !pass) e = cudaDeviceSynchronize();
    if (e == cudaSuccess && !pass && value_side) {
      L->d_usum = reinterpret_cast<float*>(base + o_usum);
      e = compute_usum(L, L->d_usum);
    }
    if (e == cudaSuccess && pad_theta) { L->theta_rows = base + o_theta; e = pad_params(desc->theta, base + o_theta, (long long)rows, desc->n, np, nullptr); }
    if (e == cudaSuccess && pad_U) { L->U_rows = base + o_U; e = pad_params(desc->U, base + o_U, (long long)rows, desc->n, np, nullptr); }
    if (e == cudaSuccess && !pass) e = cudaDeviceSynchronize();
  }
  if (e != cudaSuccess) {
    if (L->d_block) cudaFree(L->d_block);
    map_cache_destroy(L->maps);
    delete L;
    return cuda_status(e);
  }
  *out = L;
  return KVC_OK;
}

int kvc_layer_destroy(kvc_layer* L) {
  if (!L) return KVC_OK;
  if (L->d_block) cudaFree(L->d_block);
  map_cache_destroy(L->maps);
  delete L;
  return KVC_OK;
}

int kvc_layer_capsules_written(kvc_layer* L) {
  if (!L) return KVC_ERR_ARG;
  L->capsules_fresh = 1;
  return KVC_OK;
}

int kvc_layer_m(const kvc_layer* L) { return L ? L->m : -1; }

int kvc_layer_rows(const kvc_layer* L, int* key_rows, int* value_rows) {
  if (!L) return KVC_ERR_ARG;
  if (key_rows) *key_rows = L->mk;
  if (value_rows) *value_rows = L->mv;
  return KVC_OK;
}

// bytes of the key part of a capsule store (the value part follows it)
static size_t key_part_bytes(const kvc_layer* L, int B, int R) {
  return (size_t)B * L->desc.H_kv * R * L->mk * D * elem_bytes(L->desc.dtype);
}

size_t kvc_capsule_bytes(const kvc_layer* L, int B, int R) {
  if (!L || B < 0 || R < 0) return 0;
  return (size_t)B * L->desc.H_kv * R * ((size_t)L->mk + L->mv) * D * elem_bytes(L->desc.dtype);
}

size_t kvc_workspace_bytes(const kvc_layer* L, int B, int R, int T_cap) {
  if (!L || B < 0 || R < 0 || T_cap < 0) return 0;
  const size_t phases = ws_layout(L, B, R, T_cap, WS_UNIFORM | WS_RAGGED).total, cluster = cluster_ws_bytes(L, B, R, T_cap);
  size_t most = phases > cluster ? phases : cluster;
  if (B > 0 && R > 0) most = std::max(most, std::max(spread_ws_bytes(L, B, R), spread_f32_ws_bytes(L, B, R)));
  const size_t plain = (R == 0 || L->passthrough) && L->desc.dtype == KVC_BF16 && B > 0 ? plain_ws(L, B).bytes : 0;
  return most > plain ? most : plain;
}

int kvc_compress(const kvc_layer* L, const void* K_vis, const void* V_vis, int B, int R, void* capsules,
                 void* stream) {
  if (!L || B < 0 || R < 0) return KVC_ERR_ARG;
  if (B == 0 || R == 0) return KVC_OK;
  if (!K_vis || !V_vis || !capsules) return KVC_ERR_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const size_t kbytes = key_part_bytes(L, B, R), vbytes = kvc_capsule_bytes(L, B, R) - kbytes;
  void* Kc = capsules;
  void* Vc = static_cast<char*>(capsules) + kbytes;
  const_cast<kvc_layer*>(L)->capsules_fresh = 1;
  // a side kept verbatim (rho = 0, or the one-sided modes) is a plain copy of its n rows per block
  const bool k_copy = L->passthrough || L->mode == KVC_MODE_V_ONLY, v_copy = L->passthrough || L->mode == KVC_MODE_K_ONLY;
  bool used = false;
  cudaError_t e = cudaSuccess;
  if (!k_copy || !v_copy)       // bf16: both compressed sides in one kernel, which clears the status word of this call
    e = launch_compress_tc(L, K_vis, V_vis, B, R, (long long)R * L->desc.n, k_copy ? 0 : 1, v_copy ? 0 : 1, Kc, Vc, nullptr, st, &used);
  if (e == cudaSuccess && !used) e = cudaMemsetAsync(L->d_cstatus, 0, sizeof(int), st);
  if (e == cudaSuccess && k_copy) e = cudaMemcpyAsync(Kc, K_vis, kbytes, cudaMemcpyDeviceToDevice, st);
  if (e == cudaSuccess && !k_copy && !used) e = launch_compress_keys(L, K_vis, B, R, Kc, st);
  if (e == cudaSuccess && v_copy) e = cudaMemcpyAsync(Vc, V_vis, vbytes, cudaMemcpyDeviceToDevice, st);
  if (e == cudaSuccess && !v_copy && !used) e = launch_compress_values(L, V_vis, B, R, Vc, st);
  return cuda_status(e);
}

}  // extern "C"

namespace kvc {
// Which bf16 shapes take the three-kernel path (the others take the one-kernel path).  Measured on B200 over batch 1-64,
// 2-32 blocks and ratios 0.2-0.8 at n = 1024, G = 7: ahead of the one-kernel variants at 31 of 33 points (by 1.0-2.1 x;
// behind by at most 12 % at ratio 0.8 with few rows); behind them for short blocks (n = 256: 35 vs 21 us, n = 576: 74 vs
// 41 us at the 7B shapes), where the logits of a unit fit the registers of the one-kernel path.
// KVC_EXPANSION=split forces it where its plan applies, any other value of the variable keeps it off.
static bool use_split(const kvc_layer* L, int B, int R) {
  if (L->use_tc != 3 && !(L->use_tc == 0 && L->desc.n > 640)) return false;
  return plan_split(L, B, R).ok != 0;
}

constexpr double HBM_US = 6.5e6;      // bytes a microsecond at the measured copy bandwidth, in the estimates below

// Which calls with per-sequence lengths and n a multiple of 64 take the one-kernel path (1), which the cluster path (2), which the
// three-phase kernels (0).  The one-kernel path's time goes with the rounds of its units over the SMs (a unit: 9 us and 0.09 us per retained
// row, or its bytes, parameters included, at 45 GB/s, up to 90 where few units of long blocks share the L2); the three-phase kernels'
// with the bytes and the block length; the cluster path's is a chain of some 28 us, long for text, but it spreads few blocks over more SMs.
// Measured on B200, us per call, one-kernel / cluster / three-phase:
// One query head per KV head: 8 x 5 blocks of n = 576, 512 text rows 43.9 / 75.1 / 70.2; 8 x 4 of 1024 76 / 97 / 116; 1 x 5 of 576 29.1 /
// 31.1 / 31.3; 32 x 5 of 576 147 / 205 / 183; 64 x 1 of 576 194 / 148 / 123; 24 x 1 of 1024 136 / 104 / 118.
// Groups of query heads, units within one round: 16 x 2 of 1024, 32/8 heads, 80 MB of rows 47 / 58 / 79, 16 x 2 of 576 31 / 41 / 48, 6 x 8 of
// 320, m = 128, 25 / 30 / 34, but 2 x 2 of 576, 4 MB, 28 / 25 / 29, 4 x 4 of 1024, 28/4 heads, 49 / 37 / 72; more rounds: 16 x 5 of 576,
// 28/4 heads 63 / 39 / 102.
static int ragged_path(const kvc_layer* L, int B, int R, int T) {
  if (L->mode != KVC_MODE_KV || L->passthrough || R < 1 || (L->use_tc != 0 && L->use_tc != -1)) return 0;
  const FusedPlan f = plan_fused(L, B, R, true);
  if (L->use_tc == -1) return f.ok;
  const int sms = L->num_sms > 0 ? L->num_sms : 148, n = L->desc.n, m = L->m, H = L->desc.H_kv;
  const double rows = 512.0 * B * R * H * m, text = 512.0 * B * H * (double)T, par = 4.0 * m * n;
  if (L->G > 1) return f.ok && f.units <= sms && (m <= 144 || rows >= 2.5e7) ? 1 : 2;
  const double floor_us = (rows + text + H * par) / HBM_US, phases = 8.0 + 0.042 * n + 1.3 * floor_us;
  const ClusterPlan c = plan_cluster(L, B, R, T, true);
  const double cluster = c.ok && c.units <= c.ucl ? 28.0 + (n > 576 ? 0.06 * (n - 576) : 0.0) + (1.15 * (rows + H * par) + 2.5 * text) / HBM_US : 1e30;
  double fused = 1e30;
  if (f.ok) {
    const int last = (f.units + sms - 1) / sms, ctas = f.units < sms ? f.units : sms;
    const double rate = n <= 640 || sms * 45 > 90 * ctas ? (n <= 640 ? 45e3 : 90e3) : 45e3 * sms / ctas;
    const double rounds = last > 1 ? 0.5 * ((double)f.units / sms + last) : 1.0;
    fused = std::max(last * (9.0 + 0.09 * m), rounds * ((rows + text) / f.units + par) / rate);
  }
  if (fused < 0.95 * std::min(phases, cluster)) return 1;
  return cluster < 0.9 * phases ? 2 : 0;
}

// Few query heads per KV head, expansions in fp32 where the three-phase kernels make them: whether those are ahead of the cluster path.  The
// cluster path's time goes with the rounds of its units (18 us each, and its tiles, sequences and row chunks), the three-phase kernels'
// with the chunks of 64 positions of 16 expansion rows, the retained rows they walk, and the bytes.  Constants fitted (least squares of the
// relative error: 8 % and 12 %) to 1620 uniform calls on B200: 1/1 to 32/32 and 8/2, 32/8 heads, 1 x 1 to 64 x 2 blocks of n = 81 to 961, m = 11
// to 769, 0 to 700 text rows; routed by it the calls take 0.6 % more than each on its better path, and 16 of 2430 more than 10 %
// over what the three-phase kernels took before there was a cluster path (at worst 20.0 for 16.3).
// us per call, cluster / three-phase: 16/16 heads, 64 x 2 of n = 81, m = 11, 60 text rows 78 / 33; 32/32, 7 x 2 of 529, m = 67 53 / 31, m = 424 92 / 107; 4/4, 64 x 2 of 81, 700 rows 85 / 50; 8/2, 16 x 5 of 729, m = 292 45 / 143.
static bool cuda_core_expansion_wins(const kvc_layer* L, int B, int R, int T, bool ragged) {
  const ClusterPlan c = plan_cluster(L, B, R, T, ragged);
  if (!c.ok) return true;
  const int n = L->desc.n, m = L->m, H = L->desc.H_kv, nb = B * R;
  const double rows = 512.0 * nb * H * (double)m, text = 512.0 * B * H * (double)T;
  const double rounds = (c.units + c.ucl - 1) / c.ucl, rb = ceil_div(nb, c.units / H), seqs = std::min(rb, rb / R + (R > 1 && rb > 1 ? 1.0 : 0.0));
  const double cluster = rounds * (18.0 + (0.6 * rb * c.vt + 0.44 * seqs) / c.NS + 1.4 * c.nk1) - 2.0 + (rows + 4.0 * H * m * n + 1.2 * text) / HBM_US;
  const WsLayout w = ws_layout(L, B, R, T);
  const double walk = w.IR / EXP_IC, chunks = (double)H * ceil_div(nb * L->G, EXP_ROWS) * ceil_div(n, EXP_IC);
  const double phases = 15.7 + walk * (0.063 * m - 2.5) + chunks * (2.24e-4 * m + 0.0132) + (1.7 * rows + 1.57 * text) / HBM_US + 1.35 * (L->G - 1) + c.nk1;
  return phases < cluster;
}

// Which bf16 shapes take the cluster path.  Measured on B200, us per call, cluster / other paths.
// Block lengths that are no multiple of 64, and per-sequence lengths outside the path above: the other way is the three-phase kernels.
// Where those expand on the CUDA cores (n no multiple of 8) it is ahead from seven query heads per KV head on (8 x 5 blocks of n = 729,
// 28/4 heads: 37 / 277); below, by the estimate above (cuda_core_expansion_wins).  And it is ahead, with more than one query head per KV
// head, where they expand on mma.sync (4 x 1 of 400: 22 / 29; 16 x 4 of 196, 32/8 heads: 31 / 65; 1 x 1 of 784, 8/2 heads: 23 / 25; 8 x 2 of 144: 18.8 / 18.6; with lengths per sequence from 1e7 flop of expansion on: 8 x 5 of
// 144, 6/2 heads, 8e6: 21.7 / 20.8; 2 x 5 of 144, 28/4 heads, 9e6: 22 / 27); with one, its 128-row tiles stay empty (8 x 4 of 400, 32/32
// heads: 60 / 50).
// Whole multiples of 64 up to 640, groups of query heads: the other way is the one-kernel path, whose time goes with the rounds of its
// units and the retained rows (9 us + 0.09 us a row).  The cluster path is ahead (a) on the smallest calls, one unit per KV head, from m
// = 224 on (1 x 1 of n = 576, 28/4 heads: 22.0 / 24.8; n = 640: 22 / 26; m = 205: 21.6 / 20.0), (b) where the rounds of the other are many
// and its own units are one wave or fill the last (16 x 5 of 576: 43 / 57; 8 x 16 of 640: 49 / 62; 16 x 20 of 576, 16/2 heads: 53 / 88; 64
// x 8 of 576: 169 / 193; but 32 x 8 of 576, 32/8 heads, 290 MB: 151 / 114).
// KVC_EXPANSION=cluster forces it where its plan applies, any other value of the variable keeps it off.
static bool use_cluster(const kvc_layer* L, int B, int R, int T, bool ragged) {
  if (R < 1 || L->passthrough || L->mode != KVC_MODE_KV || L->desc.dtype != KVC_BF16) return false;
  if (L->use_tc == 5) return true;
  const int n = L->desc.n, G = L->G;
  if (L->use_tc != 0 || n < 64) return false;
  if (ragged || n % 64 != 0) {
    if (ragged && (n == 64 || n == 128 || n == 192 || n == 256) && plan_resident(L, B, R, 0).ok) return false;     // read the lengths itself
    if (ragged && n % 64 == 0 && n <= 1024 && cluster_terms(L) == 1) {
      const int path = ragged_path(L, B, R, T);
      if (path != 2 || G == 1) return path == 2;
    }
    if (cluster_terms(L) == 2) return G > 4 || !cuda_core_expansion_wins(L, B, R, T, ragged);
    return G > 1 && (!ragged || 4.0 * B * L->desc.H_q * R * (double)L->m * n >= 1e7);
  }
  if (n <= 256 || n > 640 || G == 1) return false;
  const int sms = L->num_sms > 0 ? L->num_sms : 148;
  const double rows = 512.0 * B * R * L->desc.H_kv * L->m, bytes = rows + 512.0 * B * L->desc.H_kv * (double)T;
  if (B * R * (long long)G <= 64) return bytes < 8e6 && L->m >= 224;
  const FusedPlan f = plan_fused(L, B, R);
  if (f.ok && f.units <= sms) return false;
  const ClusterPlan c = plan_cluster(L, B, R, T, false);
  if (!f.ok || !c.ok) return c.ok != 0;
  const int rounds = (c.units + c.ucl - 1) / c.ucl;
  if (10ll * c.units < 7ll * rounds * c.ucl) return false;
  return 1.1 * (25.0 * rounds + 4.0 + 2.4 * bytes / HBM_US) < (f.units + sms - 1) / sms * (9.0 + 0.09 * L->m);
}

// Which bf16 shapes take the spread path: those its plan serves (at most 64 expansion rows per group of blocks, clusters of two or more CTAs for
// all groups at once, scores and weights that leave room for a ring).  Over 110 drawn calls of that kind (1/1 to 32/32 heads, n = 64 to 1024, up
// to 3000 text rows) it took 14.4 us in the geometric mean, the paths below 23.8; behind them are:
// short blocks whose parameters the resident path keeps in shared memory, with more than two row tiles (5 x 9 of n = 256, 28/4 heads 13.4 / 12.5;
// 2 x 8 13.2 / 11.0; but 2 x 2 8.8 / 10.3, 1 x 1 9.0 / 10.8), few retained rows (5 x 1, m = 32, 16/2 heads 8.4 / 7.6; 4 x 4, m = 52, 8/2 heads
// 8.6 / 8.7), long text (1 x 2, 4096 rows 14.8 / 12.3; 4 x 2, 1024 rows, 10.1 / 13.1) or n = 64 (8.8 / 8.3); and the longest chains beside the
// one-kernel and three-kernel paths (3 x 13 of 1024, 28/4 heads 48.3, estimated 39.4, / 41.1; 14 x 16 of 256, m = 167, 16/2 heads 23.9 / 23.2).
// Calls whose path the tests name stay where they are, although this one is ahead: lengths per sequence on those short
// blocks (6 x 1 of n = 256, 8/2 heads 10.3 / 13.4) or under 1e7 flop of expansion beside them, and clusters of two on blocks under 96 positions
// (32 x 1 of n = 81, 8/2 heads, 700 rows 12.3 / 36.9).  KVC_EXPANSION=spread forces it where its plan applies, any other value keeps it off.
// More than eight query heads per KV head: where its estimate is ahead of one of the path it stands before.  Of 881 drawn calls with 9 to 16
// it is the faster path for 662; taken for all that the rules above give it, 145 were more than 3 % longer, at worst 2.1 times (13 x 12 of 1024,
// 10/1 heads 61 / 34; 9 x 11 of 256, 28/2 heads, 1492 rows 32 / 22); by the estimates about 30, at worst 1.3 times, and the geometric mean of all
// is 0.79 of the other paths' time (0.82 before; 0.78 with every call on its better path).
// The cluster path: rounds of units and their tiles, the bytes; fitted to 97 uniform calls of up to eight query heads per KV head, 10 %
static double cluster_estimate(const kvc_layer* L, int B, int R, int T, int terms) {
  const int n = L->desc.n, m = L->m, H = L->desc.H_kv, sms = L->num_sms > 0 ? L->num_sms : 148;
  const int units = H * ceil_div(B * R, CL_ROWS / L->G), NS = ceil_div(ceil_div(n, 64), terms == 2 ? 2 : 4);
  const int held = sms * 88 / 100 / NS, rounds = ceil_div(units, held > 0 ? held : 1);
  const double rows = 512.0 * B * R * H * (double)m + 4.0 * H * (double)m * n, text = 512.0 * B * H * (double)T;
  return rounds * (24.4 + 1.93 * ceil_div(m, 64)) - 4.2 + (1.71 * rows + 1.86 * text) / HBM_US + 0.0137 * B * H;
}
// The path a call with more than eight query heads per KV head would take otherwise: fitted (least squares of the relative error) to those calls,
// the one-kernel path's 10 %, the three-kernel path's 13 %, the cluster path's as above and 14 % too short for them.  Blocks longer than its
// clusters hold go to the three-phase kernels, which the spread path is always ahead of there (2 x 2 of n = 1444, 48/4 heads 57 / 161).
static double general_estimate(const kvc_layer* L, int B, int R, int T, bool ragged, int terms) {
  const int n = L->desc.n, m = L->m, H = L->desc.H_kv, sms = L->num_sms > 0 ? L->num_sms : 148;
  const double cluster = ceil_div(ceil_div(n, 64), terms == 2 ? 2 : 4) <= CL_MAX_NS ? 1.1 * cluster_estimate(L, B, R, T, terms) : 1e30;
  if (n % 64 != 0 || (ragged && ragged_path(L, B, R, T) != 1)) return cluster;
  if (!ragged && n > 640 && plan_split(L, B, R).ok)
    return 1.05 * (16.2 + 0.0214 * m + 0.124 * H * ceil_div(B * R * L->G, 128) + 2.0 * 512.0 * B * H * (2.0 * R * m + 2.0 * T) / HBM_US + 3.5e-4 * H * n);
  double fused = 1e30;
  const FusedPlan f = plan_fused(L, B, R, ragged);
  if (f.ok) {
    const int waves = ceil_div(f.units, sms);
    const double text = (double)T / f.nrg;                   // of a unit, shared by the warps that its blocks' columns occupy
    fused = 9.4 + 0.0346 * m + 16.1 * (waves - 1) + 7.2e-5 * waves * m * (double)n + 4.96e-3 * text + 35e-3 * text / (ceil_div(R, f.nrg) * (n / 64)) +
            (f.nrg > 1 ? 4.9 : 0.0);
  }
  return ragged || n <= 256 || n > 640 ? fused : std::min(fused, cluster);
}
static bool use_spread(const kvc_layer* L, int B, int R, int T, bool ragged, const SpreadPlan& p) {
  if (!p.ok || L->use_tc == 6) return p.ok != 0;
  const int n = L->desc.n;
  if (plan_resident(L, B, R, T).ok) return !ragged && n == 256 && L->m > 48 && R * L->G <= 16 && T <= 128 * p.C;
  if (ragged && n % 8 == 0 && n % 64 != 0 && 4.0 * B * L->desc.H_q * R * (double)L->m * n < 1e7) return false;
  if (n % 64 == 0 && p.us > (L->G > 8 ? (n > 640 ? 42.0 : 1e30) : (n <= 256 ? 24.0 : 36.0))) return false;
  if (L->G > 8 && p.waves == 1) return p.us < general_estimate(L, B, R, T, ragged, p.terms);
  // several waves: where it is ahead of the estimate of the cluster path.  Routed by it those take 0.89 of their time before in the geometric mean,
  // none more than 3 % longer (16 x 8 of n = 144, 28/4 heads, 715 rows 16.5 / 32.3; 25 x 5 of 400, 1610 rows 46 / 89; 8 x 7 of 324, 32/32 heads
  // 74 / 88; not: 26 x 10 of 121 45 / 34)
  if (p.waves > 1) return !ragged && n >= 96 && p.us < 0.85 * cluster_estimate(L, B, R, T, p.terms);
  return n >= 96 || p.C * p.nrg > 2;
}

// Which fp32 calls take the spread path (410 of 492 drawn ones, half the three-phase kernels' time in the geometric mean; three of them are longer than
// there, with one query head per KV head and many retained rows, at worst 2 x 2 of n = 729, m = 438, 32/32 heads, 158 / 138, which neither
// estimate tells apart): those of one wave of clusters (0.29 to 0.97 of the three-phase kernels' time over 44 drawn calls), and
// of up to four where its estimate is under nine tenths of theirs (0.74 with lengths per sequence, whose sum it does not see: 11 x 4 of n = 841,
// 28/4 heads, 316, estimated 268 to 359, / 299; 0.7 with one query head per KV head: 2 x 3 of 1024, 32/32 heads 250,
// estimated 199, / 194; 13 x 3 of 169, 28/4 heads 52 / 97; 16 x 8 of 169 95 / 128).  Their estimate: the columns and chunks of a CTA's walk,
// the waves of CTAs and the bytes, fitted to the same 70 shapes (16 %).
// Calls with lengths per sequence of less than 3e7 flop of expansion stay on the three-phase kernels, whose path the tests name.
static bool use_spread_f32(const kvc_layer* L, int B, int R, int T, bool ragged, const SpreadPlan& p) {
  if (!p.ok || L->use_tc == 6) return p.ok != 0;
  const int n = L->desc.n, m = L->m, H = L->desc.H_kv;
  if (ragged && 4.0 * B * L->desc.H_q * R * (double)m * n < 3e7) return false;
  if (p.waves <= 1) return true;
  const WsLayout w = ws_layout(L, B, R, T);
  const double tiles = (double)H * ceil_div(B * R * L->G, EXP_ROWS), walk = (double)(w.IR / EXP_IC) * m;
  const double phases = 9.7 + 0.0466 * walk + 0.0251 * std::ceil(tiles * w.NS / 296.0) * walk + 2.03e-4 * tiles * ceil_div(n, EXP_IC) * m +
                        3.14 * 2.0 * H * ((double)B * R * m + (double)B * T) * 512.0 / HBM_US + 4.46 * L->G + 0.0423 * R * B * H;
  return p.us < (L->G == 1 ? 0.7 : (ragged ? 0.74 : 0.9)) * phases;
}

// One token per decode call, process-wide: never 0 and never one of the byte patterns a caller is likely to have
// filled a fresh workspace with, so that stale workspace contents cannot pass for arrivals of this call.
static unsigned int next_token() {
  static std::atomic<unsigned int> counter{0x1000u};
  for (;;) {
    const unsigned int t = counter.fetch_add(1u, std::memory_order_relaxed) + 1u;
    const unsigned int b0 = t & 0xffu;
    const bool uniform = ((t >> 8) & 0xffu) == b0 && ((t >> 16) & 0xffu) == b0 && (t >> 24) == b0;
    if (t != 0u && !uniform) return t;
  }
}

int decode_common(const kvc_layer* L, const void* q, const void* capsules, int B, int R, const void* K_txt,
                  const void* V_txt, int T, int T_cap, void* out, void* workspace, cudaStream_t st, const int* R_b,
                  const int* T_b, size_t ws_limit) {
  if (!L || B < 0 || R < 0 || T < 0 || T_cap < T) return KVC_ERR_ARG;
  if (B == 0) return KVC_OK;
  if (R == 0 && T == 0) return KVC_ERR_SHAPE;
  if (!q || !out || (R > 0 && !capsules) || (T > 0 && (!K_txt || !V_txt))) return KVC_ERR_ARG;
  if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255)) return KVC_ERR_WORKSPACE;

  DecodeArgs a{};
  char* ws = static_cast<char*>(workspace);
  a.q = q;
  a.Kc = capsules;
  a.Vc = capsules ? static_cast<const char*>(capsules) + key_part_bytes(L, B, R) : nullptr;
  a.K_txt = K_txt; a.V_txt = V_txt;
  a.theta = L->desc.theta; a.U = L->desc.U; a.mu = L->desc.mu;
  a.out = out;
  a.B = B; a.H_kv = L->desc.H_kv; a.G = L->G; a.R = R; a.m = L->mk; a.ms = (L->mk + 15) / 16 * 16; a.n = L->desc.n;
  a.mv = L->mv; a.msv = (L->mv + 15) / 16 * 16;
  a.id_theta = L->mode == KVC_MODE_V_ONLY; a.id_U = L->mode == KVC_MODE_K_ONLY;
  a.T = T; a.T_cap = T_cap > 0 ? T_cap : 1;
  a.passthrough = L->passthrough;
  a.token = next_token();
  a.cnt = reinterpret_cast<int*>(ws);                       // counters and the status word lead the workspace on every path
  a.status = a.cnt + (size_t)B * L->desc.H_kv;
  a.R_b = R_b; a.T_b = T_b;
  a.early_capsules = L->capsules_fresh ? 0 : 1;
  const_cast<kvc_layer*>(L)->capsules_fresh = 0;
  const bool ragged = R_b != nullptr || T_b != nullptr;
  const uintptr_t align = reinterpret_cast<uintptr_t>(q) | reinterpret_cast<uintptr_t>(capsules) |
                          reinterpret_cast<uintptr_t>(out) | (T > 0 ? reinterpret_cast<uintptr_t>(K_txt) |
                          reinterpret_cast<uintptr_t>(V_txt) : 0) | reinterpret_cast<uintptr_t>(L->desc.mu);

  if ((align & 15) == 0) {
    const SpreadPlan sp = plan_spread(L, B, R, T, ragged);
    if (use_spread(L, B, R, T, ragged, sp) && (ws_limit == 0 || spread_ws(L, sp, B).bytes <= ws_limit)) {
      bool encoded = false;
      const cudaError_t se = launch_spread(L, a, sp, ws, st, &encoded);
      if (encoded) return cuda_status(se);
    }
  }

  if ((align & 15) == 0) {
    const SpreadPlan sp = plan_spread_f32(L, B, R, T);
    if (use_spread_f32(L, B, R, T, ragged, sp) && (ws_limit == 0 || spread_ws(L, sp, B).bytes <= ws_limit)) return cuda_status(launch_spread_f32(L, a, sp, ws, st));
  }

  if ((align & 15) == 0 && use_cluster(L, B, R, T, ragged)) {
    const ClusterPlan cp = plan_cluster(L, B, R, T, ragged);
    if (cp.ok && (ws_limit == 0 || cluster_ws(L, cp, B).bytes <= ws_limit)) {
      bool encoded = false;
      const cudaError_t ce = launch_cluster(L, a, cp, ws, st, &encoded);
      if (encoded) return cuda_status(ce);
    }
  }

  // rows stored verbatim only (uncompressed K/V, text alone, the stores of ratio 0)
  if ((align & 15) == 0 && (R == 0 || L->passthrough) && !ragged && L->use_tc != -2) {
    const PlainPlan pp = plan_plain(L, B, R * L->desc.n, T);
    if (pp.ok && (ws_limit == 0 || plain_ws(L, B).bytes <= ws_limit)) {
      bool encoded = false;
      const cudaError_t pe = launch_plain(L, a, pp, ws, st, &encoded);
      if (encoded) return cuda_status(pe);
    }
  }

  a.ws = ws_layout(L, B, R, T, ragged ? WS_RAGGED : WS_UNIFORM);
  a.Ts = a.ws.Ts;
  a.S = reinterpret_cast<float*>(ws + a.ws.off_S);
  a.Sb = reinterpret_cast<__nv_bfloat16*>(ws + a.ws.off_S);
  a.s_txt = reinterpret_cast<float*>(ws + a.ws.off_stxt);
  a.W = reinterpret_cast<float*>(ws + a.ws.off_W);
  a.wstat = reinterpret_cast<float2*>(ws + a.ws.off_wstat);
  a.Wcomb = reinterpret_cast<float*>(ws + a.ws.off_Wc);
  a.statc = reinterpret_cast<float4*>(ws + a.ws.off_statc);
  a.ypart = reinterpret_cast<float*>(ws + a.ws.off_ypart);
  a.ystat = reinterpret_cast<float2*>(ws + a.ws.off_ystat);
  a.fcnt = reinterpret_cast<unsigned long long*>(ws + a.ws.off_fcnt);
  a.fpart_y = reinterpret_cast<float*>(ws + a.ws.off_fpy);
  a.fpart_ml = reinterpret_cast<float2*>(ws + a.ws.off_fpml);
  a.split_base = ws + a.ws.off_split;
  a.resident_base = ws + a.ws.off_resident;

  // bf16 storage with TMA-compatible shapes and pointers: the whole of Algorithm 1 in one kernel
  {
    const bool plain = R == 0 || L->passthrough;            // rows stored verbatim only: served above
    // one-sided modes are served by the three-phase kernels below
    const bool one_sided = R > 0 && L->mode != KVC_MODE_KV;
    // Short blocks whose theta and U fit shared memory (n <= 256, m <= 128, G <= 8) take the resident-parameter kernel: on
    // the n = 256, G = 7, m = 103 shape it ran ahead of the other one-kernel variants at every batch measured (1, 4, 16:
    // 19.2 / 19.5 / 42.4 us against 22.4 / 23.5 / 83.7 us).  KVC_EXPANSION=resident forces it, any other value keeps it off.
    if (!plain && L->mode == KVC_MODE_KV && (align & 15) == 0 && (L->use_tc == 4 || L->use_tc == 0)) {
      const ResidentPlan rp = plan_resident(L, B, R, T);
      if (rp.ok) {
        bool encoded = false;
        const cudaError_t re = launch_resident(L, a, rp, st, &encoded);
        if (encoded) return cuda_status(re);
      }
    }
    if (!plain && !one_sided && !ragged && (align & 15) == 0 && T <= 64 * SP_OUT_ROWS * SP_TEXT_CHUNK && use_split(L, B, R)) {
      const SplitPlan sp = plan_split(L, B, R);
      bool encoded = false;
      const cudaError_t se = launch_split(L, a, sp, st, &encoded);
      if (encoded) return cuda_status(se);
    }
    FusedPlan fp{};
    if (!plain && !one_sided && (!ragged || ragged_path(L, B, R, T) == 1)) fp = plan_fused(L, B, R, ragged);
    if (fp.ok && (align & 15) == 0) {
      bool encoded = false;
      const cudaError_t fe = launch_fused(L, a, fp, st, &encoded);
      if (encoded) return cuda_status(fe);
    }
  }

  cudaError_t e = launch_scores(a, L->desc.dtype, st);
  if (e == cudaSuccess) e = launch_expand(a, L->desc.dtype, st);
  if (e == cudaSuccess) e = launch_output(a, L->desc.dtype, st);
  return cuda_status(e);
}
}  // namespace kvc

extern "C" {

int kvc_decode_attend(const kvc_layer* L, const void* q, const void* capsules, int B, int R, const void* K_txt,
                      const void* V_txt, int T, int T_cap, void* out, void* workspace, void* stream) {
  return decode_common(L, q, capsules, B, R, K_txt, V_txt, T, T_cap, out, workspace,
                       static_cast<cudaStream_t>(stream));
}

int kvc_decode_attend_ragged(const kvc_layer* L, const void* q, const void* capsules, int B, int R_max, const int* R_b,
                             const void* K_txt, const void* V_txt, int T_max, const int* T_b, int T_cap, void* out,
                             void* workspace, void* stream) {
  return decode_common(L, q, capsules, B, R_max, K_txt, V_txt, T_max, T_cap, out, workspace,
                       static_cast<cudaStream_t>(stream), R_b, T_b);
}

int kvc_compress_ragged(const kvc_layer* L, const void* K_vis, const void* V_vis, int B, int N_cap, const int* N_v,
                        int R_max, void* capsules, void* K_tail, void* V_tail, int T_cap, int* R_b, int* T_b, void* stream) {
  if (!L || B < 0 || N_cap < 0 || R_max < 0 || T_cap < 0) return KVC_ERR_ARG;
  if (B == 0) return KVC_OK;
  if (!N_v || !R_b || !T_b || (N_cap > 0 && (!K_vis || !V_vis)) || (R_max > 0 && !capsules) ||
      (T_cap > 0 && (!K_tail || !V_tail)))
    return KVC_ERR_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const_cast<kvc_layer*>(L)->capsules_fresh = 1;
  void* Vc = capsules ? static_cast<char*>(capsules) + key_part_bytes(L, B, R_max) : nullptr;
  return cuda_status(launch_compress_ragged(L, K_vis, V_vis, B, N_cap, N_v, R_max, capsules, Vc, K_tail, V_tail, T_cap,
                                            R_b, T_b, st));
}

int kvc_attend_full(const kvc_layer* L, const void* q, const void* K, const void* V, int B, int S, int S_cap,
                    void* out, void* workspace, void* stream) {
  return decode_common(L, q, nullptr, B, 0, K, V, S, S_cap, out, workspace, static_cast<cudaStream_t>(stream));
}

int kvc_collapse_theta(const void* W1, const void* W2, int H_kv, int m, int k, int n, kvc_dtype dtype, void* theta_out,
                       void* stream) {
  if (!W1 || !W2 || !theta_out) return KVC_ERR_ARG;
  if (H_kv < 1 || m < 1 || k < 1 || n < 1 || H_kv > 65535 || (m + 63) / 64 > 65535) return KVC_ERR_SHAPE;
  if (dtype != KVC_F32 && dtype != KVC_BF16) return KVC_ERR_DTYPE;
  return cuda_status(kvc::launch_collapse_theta(W1, W2, theta_out, H_kv, m, k, n, (int)dtype, static_cast<cudaStream_t>(stream)));
}

int kvc_selftest_bounded_wait(void* stream) {
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  int* d_status = nullptr;
  cudaError_t e = cudaMalloc(&d_status, sizeof(int));
  if (e != cudaSuccess) return cuda_status(e);
  int h_status = KVC_ERR_CUDA;
  e = cudaMemsetAsync(d_status, 0, sizeof(int), st);
  if (e == cudaSuccess) {
    kvc::launch_wait_selftest(d_status, st);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(&h_status, d_status, sizeof(int), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  cudaFree(d_status);
  if (e != cudaSuccess) return cuda_status(e);
  return h_status;
}

int kvc_read_device_status(const kvc_layer* L, int B, int R, int T, const void* workspace, int* status_out) {
  if (!L || !status_out || B < 0 || R < 0 || T < 0) return KVC_ERR_ARG;
  if (!workspace) {                           // the fixed scratch array of kvc_decode_attend_static on this device
    void* p = nullptr;
    const int s = kvc::static_scratch(&p);
    if (s != KVC_OK) return s;
    workspace = p;
  }
  const WsLayout w = ws_layout(L, B, R, T);
  const char* p = static_cast<const char*>(workspace) + w.off_cnt + sizeof(int) * (size_t)B * L->desc.H_kv;
  return cudaMemcpy(status_out, p, sizeof(int), cudaMemcpyDeviceToHost) == cudaSuccess ? KVC_OK : KVC_ERR_CUDA;
}

int kvc_read_compress_status(const kvc_layer* L, int* status_out) {
  if (!L || !status_out) return KVC_ERR_ARG;
  return cudaMemcpy(status_out, L->d_cstatus, sizeof(int), cudaMemcpyDeviceToHost) == cudaSuccess ? KVC_OK : KVC_ERR_CUDA;
}

int kvc_export_maps(const kvc_layer* L, int R, int32_t* idx_out, int32_t* group_out) {
  if (!L || R < 0) return KVC_ERR_ARG;
  if (idx_out) {
    if (cudaMemcpy(idx_out, L->d_idx, (size_t)L->desc.H_kv * L->m * sizeof(int32_t), cudaMemcpyDeviceToHost) !=
        cudaSuccess)
      return KVC_ERR_CUDA;
  }
  if (group_out && R > 0) {
    // written by a kernel with the row arithmetic of the key selection (block r, offset i -> row r*n + i)
    const size_t bytes = (size_t)R * L->desc.n * 2 * sizeof(int32_t);
    int32_t* d = nullptr;
    if (cudaMalloc(&d, bytes) != cudaSuccess) return cuda_status(cudaGetLastError());
    cudaError_t e = cudaMemset(d, 0xff, bytes);
    if (e == cudaSuccess) e = kvc::launch_export_groups(d, R, L->desc.n, nullptr);
    if (e == cudaSuccess) e = cudaMemcpy(group_out, d, bytes, cudaMemcpyDeviceToHost);
    cudaFree(d);
    if (e != cudaSuccess) return cuda_status(e);
  }
  return KVC_OK;
}

}  // extern "C"
