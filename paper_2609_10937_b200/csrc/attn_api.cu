// C ABI of the fused-attention library: argument checks, closed-form plan,
// TMA tensor maps, kernel launches.  No device memory is allocated here.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <unordered_map>

#include "attn.h"
#include "attn_kernels.cuh"
#include "attn_plan_internal.h"
#include "decode_kernels.cuh"
#include "gemm.h"
#include "gemm_kernels.cuh"
#include "narrow_kernel.cuh"
#include "pipe_kernel.cuh"

namespace {

thread_local char t_cuda_error[256] = "";
thread_local int t_launch_count = 0;
thread_local int t_cluster_size = 0;   // CTAs per thread-block cluster of the last fused launch (0: no clusters)
thread_local int t_kernel = ATTN_KERNEL_NONE, t_grid = 0;   // the last launch and its CTAs
// Name and template arguments of the last launch's kernel, put together where they are asked for.
struct Instantiation {
  const char* name = "";
  int args = 0, arg[6] = {};
};
thread_local Instantiation t_instantiation;
void launched(int kernel, long long ctas, const Instantiation& inst) { t_kernel = kernel; t_grid = (int)ctas; t_instantiation = inst; }

int cuda_fail(cudaError_t e, const char* what) {
  (void)cudaGetLastError();              // reported here: the next call must not find it again
  std::snprintf(t_cuda_error, sizeof t_cuda_error, "%s: %s", what, cudaGetErrorString(e));
  return ATTN_ERR_CUDA;
}
#define ATTN_CUDA_TRY(expr)                               \
  do {                                                    \
    cudaError_t e__ = (expr);                             \
    if (e__ != cudaSuccess) return cuda_fail(e__, #expr); \
  } while (0)

// ---- driver entry point for tensor-map encoding (no link-time libcuda dependency)
using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn get_encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  });
  return fn;
}

// 3-D map over a contiguous [BH][L][d] bf16 tensor; box = (64 columns, box_rows rows, 1 head), 128-byte swizzle.
int make_tmap(CUtensorMap* m, const void* base, int BH, int L, int d, int box_rows) {
  EncodeTiledFn fn = get_encode_fn();
  if (!fn) {
    std::snprintf(t_cuda_error, sizeof t_cuda_error, "cuTensorMapEncodeTiled entry point not found");
    return ATTN_ERR_CUDA;
  }
  cuuint64_t dims[3] = {(cuuint64_t)d, (cuuint64_t)L, (cuuint64_t)BH};
  cuuint64_t strides[2] = {(cuuint64_t)d * 2, (cuuint64_t)L * (cuuint64_t)d * 2};
  cuuint32_t box[3] = {64, (cuuint32_t)box_rows, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    std::snprintf(t_cuda_error, sizeof t_cuda_error, "cuTensorMapEncodeTiled failed with CUresult %d", (int)r);
    return ATTN_ERR_CUDA;
  }
  return ATTN_OK;
}

// ---- per-device state: workspace registry and cached descriptor
constexpr int kMaxDevices = 64;
struct DeviceState {
  void* ws = nullptr;
  size_t ws_bytes = 0;
  bool arch_checked = false;
  bool arch_ok = false;
  attn_hw_desc desc;
  int decode_clusters[5] = {};   // [i]: clusters of 2^i CTAs of the decode kernel that fit at once, + 1 (0 = not asked yet); guarded by g_mu
  int resident[2][9] = {};     // [causal][k]: clusters of k CTAs that fit at once, + 1 (0 = not asked yet); guarded by g_mu
};
DeviceState g_dev[kMaxDevices];
std::mutex g_mu;

int device_state(DeviceState** out) {
  int dev = 0;
  ATTN_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) return ATTN_ERR_INVALID_ARG;
  std::lock_guard<std::mutex> lk(g_mu);
  DeviceState& s = g_dev[dev];
  if (!s.arch_checked) {
    int rc = attn_hw_desc_query(dev, &s.desc);
    if (rc == ATTN_ERR_CUDA) return rc;
    s.arch_ok = (rc == ATTN_OK);
    s.arch_checked = true;
  }
  *out = &s;
  return s.arch_ok ? ATTN_OK : ATTN_ERR_WRONG_ARCH;
}

// Number of the current context, unlike any other of the process; 0 if none is current yet.
unsigned long long current_context() {
  using GetIdFn = CUresult (*)(CUcontext, unsigned long long*);
  static const GetIdFn fn = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuCtxGetId", &p, cudaEnableDefault, &q) != cudaSuccess || q != cudaDriverEntryPointSuccess) p = nullptr;
    return reinterpret_cast<GetIdFn>(p);
  }();
  unsigned long long id = 0;
  return fn && fn(nullptr, &id) == CUDA_SUCCESS ? id : 0;
}

// Dynamic shared memory a kernel may use, raised when a launch needs more than the last one that raised it (asking the driver
// every time took about as long as the launch itself).  The allowance belongs to the context: it is asked for again in a
// context other than the one it was last asked for in (several contexts on a device; cudaDeviceReset).
int allow_smem(const void* kern, int bytes) {
  struct Allowed { unsigned long long context; int bytes; };
  static std::mutex mu;
  static std::unordered_map<const void*, Allowed> allowed;
  const unsigned long long context = current_context();
  std::lock_guard<std::mutex> lk(mu);
  Allowed& have = allowed[kern];
  if (context != 0 && have.context == context && have.bytes >= bytes) return ATTN_OK;
  ATTN_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
  have = {context, bytes};
  return ATTN_OK;
}
#define ATTN_ALLOW_SMEM(kern, bytes)                                                 \
  do {                                                                               \
    const int rc__ = allow_smem(reinterpret_cast<const void*>(kern), bytes);         \
    if (rc__ != ATTN_OK) return rc__;                                                \
  } while (0)

// Launches a kernel whose CTAs may start while the grid in front of it on the stream is still finishing (its set-up then runs under
// that grid's last CTAs; every kernel here waits for the grids in front before it touches memory, ptx_sm100.cuh).  cluster: CTAs
// of a thread-block cluster, 0 or 1 for none.
template <class... P, class... A>
cudaError_t launch_kernel(void (*kern)(P...), long long grid, int block, int smem, int cluster, cudaStream_t stream, const A&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)cluster;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

bool overlaps(const void* a, size_t na, const void* b, size_t nb) {
  const uintptr_t a0 = (uintptr_t)a, b0 = (uintptr_t)b;
  return a0 < b0 + nb && b0 < a0 + na;
}

int check_args(const void* q, const void* k, const void* v, const void* o, int B, int H, int L, int d, int Lk = 0) {
  if (Lk == 0) Lk = L;
  if (!q || !k || !v || !o || B <= 0 || H <= 0 || L <= 0 || Lk <= 0 || d <= 0) return ATTN_ERR_INVALID_ARG;
  if (d != 64 && d != 128) return ATTN_ERR_UNSUPPORTED_SHAPE;
  if ((long long)B * H * ((L + 127) / 128) > 0x3FFFFFFFLL) return ATTN_ERR_UNSUPPORTED_SHAPE;  // grid index range
  if (((uintptr_t)q | (uintptr_t)k | (uintptr_t)v | (uintptr_t)o) & 15u) return ATTN_ERR_MISALIGNED;
  if ((long long)B * H * ((Lk + 127) / 128) > 0x3FFFFFFFLL) return ATTN_ERR_UNSUPPORTED_SHAPE;
  const size_t bytes = (size_t)B * H * L * d * 2, kv_bytes = (size_t)B * H * Lk * d * 2;
  if (overlaps(o, bytes, q, bytes) || overlaps(o, bytes, k, kv_bytes) || overlaps(o, bytes, v, kv_bytes))
    return ATTN_ERR_ALIASING;
  return ATTN_OK;
}

template <int D, int TKV, int NQ>
int launch_fwd(const void* q, const void* k, const void* v, void* o, int B, int H, int L, int Lk, const attn_tiles& t,
               float* ws, unsigned int* status, DeviceState* st, cudaStream_t stream, bool may_overlap) {
  using SM = attn::FwdSmem<D, TKV, NQ>;
  const int BH = B * H;
  CUtensorMap tq, tk, tv, to;
  int rc;
  if ((rc = make_tmap(&tq, q, BH, L, D, attn::kSub)) != ATTN_OK) return rc;
  if ((rc = make_tmap(&tk, k, BH, Lk, D, TKV)) != ATTN_OK) return rc;
  if ((rc = make_tmap(&tv, v, BH, Lk, D, TKV)) != ATTN_OK) return rc;
  if ((rc = make_tmap(&to, o, BH, L, D, 32)) != ATTN_OK) return rc;    // every warp stores its own 32 rows

  attn::FwdParams p;
  p.L = Lk;                                                       // keys per head (L: query rows per head)
  p.q_tiles = (L + NQ * attn::kSub - 1) / (NQ * attn::kSub);
  p.n_steps = (Lk + TKV - 1) / TKV;
  p.tiles = BH * p.q_tiles;
  p.stages = t.kv_stages;
  p.causal = t.causal ? 1 : 0;
  p.ratio = NQ * attn::kSub / TKV;
  p.head_units = attn::tile_prefix(p.n_steps, p.ratio, p.causal, p.q_tiles);
  p.scale_log2 = (float)(1.4426950408889634 / std::sqrt((double)D));
  p.o = reinterpret_cast<__nv_bfloat16*>(o);
  p.status = status;
  p.counters = reinterpret_cast<unsigned int*>(ws);                   // head of the workspace
  p.ws = ws ? ws + attn::kCounterBytes / sizeof(float) : nullptr;    // partial results follow
  int grid = t.ctas;
  p.seg_skip = 0;
  // One CTA per tile with more tiles than SMs: a persistent grid of one CTA per SM runs them in the same order.  (Of the device's own plans those
  // at d = 64 that pipe_tiles leaves here; at d = 128 overrides and callers' descriptors only.)
  const int sms = st->desc.num_units;                      // of the device itself (the plan may be for a smaller machine)
  if (!p.causal && t.ctas == t.tiles) {
    if (sms > 0 && t.tiles > sms) {
      grid = sms;
      p.seg_skip = (long long)(grid - 1) * p.n_steps;
    }
  }
  const long long total_units = p.head_units * BH;
  // at least one KV step per CTA; when Q tiles are shared, the counters of every (CTA, sub-tile, warp) --
  // two each -- must fit the counter block
  if (grid < 1 || (long long)grid > total_units) return ATTN_ERR_BAD_TILES;
  if (ws && (size_t)grid * NQ * 8 > attn::kCounterBytes / sizeof(unsigned int)) return ATTN_ERR_BAD_TILES;
  const int smem = SM::total(t.kv_stages);
  // uniform key split (k CTAs per tile, all parts of a tile finish together): the instantiation with fixed merge roles.
  // Its merging warps wait for the other CTAs of their tile, so every CTA of the grid must be resident at once (one
  // CTA per SM); a larger grid takes the instantiation in which the last CTA to finish merges and nobody waits for a
  // CTA that has not started.  The same holds for a launch that may run beside another one of its kind on the same
  // device (attn_forward_ws: two such kernels could each hold part of the SMs and wait for CTAs that cannot start);
  // thread-block clusters are scheduled as a whole and stay in use there.
  const bool eager = !p.causal && t.ctas > t.tiles && t.ctas % t.tiles == 0 && grid <= sms;
  const bool wait_roles_ok = !may_overlap;
  auto launch = [&](auto kern) -> int {
    ATTN_ALLOW_SMEM(kern, smem);
    ATTN_CUDA_TRY(launch_kernel(kern, grid, 512, smem, 0, stream, tq, tk, tv, to, p));
    return ATTN_OK;
  };
  // Uniform key split with few parts: the k CTAs of a tile are launched as one thread-block cluster and exchange
  // their partial results through distributed shared memory (landing areas in the K/V ring: the groups of rows one
  // CTA merges, times the k-1 parts it receives for each, must fit).  Used only if all clusters can be resident at
  // once, like the CTAs of the plain launch; otherwise, or if the cluster launch is not possible, the partials go
  // through the workspace.
  p.cluster_k = 0;
  // CTAs of the next grid that come in early take the SMs that this one leaves free, in the order in which it leaves them, and
  // where a call's time hangs on which SMs hold which CTAs that can cost more than it saves.  Early / when the CTAs end (us, graphs
  // of 12 calls): one CTA per tile on less than three quarters of the SMs, d = 128, 10 heads x 2048 33.9 / 32.9, 8 x 2500 41.4 / 39.9
  // (but 40 x 512 15.4 / 16.4, and 12 x 2000 at d = 64 the same); causal tiles cut over the whole machine 2 x 6144 45.6 /
  // 42.8, 3 x 6144 50.8 / 49.8; few rows against many keys 8 x (24 x 16384) 60.0 / 56.7.  Elsewhere early: clusters (0.95 times), waves
  // of whole tiles (0.98), other tiles cut over the machine (median 0.995; 128 x 900 85.2 / 88.7, but 64 x 1700 103 / 99).
  p.release_early = t.ctas == t.tiles ? NQ == 1 || 4 * grid >= 3 * sms || t.cost_steps < (D == 64 ? 20 : 12)
                    : p.causal        ? grid < sms
                                      : NQ == 2 || t.cost_steps < 15;
  t_cluster_size = 0;
  auto launch_eager = [&](auto kern, auto kern_cluster) -> int {
    ATTN_ALLOW_SMEM(kern, smem);
    ATTN_ALLOW_SMEM(kern_cluster, smem);
    const int kk = t.ctas / t.tiles;
    const size_t landing = (size_t)((4 * NQ + kk - 1) / kk) * (kk - 1) * (32 * D * 4 + 256);
    if (kk >= 2 && kk <= 8 && landing <= (size_t)t.kv_stages * SM::kStageBytes) {
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(grid);
      cfg.blockDim = dim3(512);
      cfg.dynamicSmemBytes = smem;
      cfg.stream = stream;
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = kk;
      attr[0].val.clusterDim.y = 1;
      attr[0].val.clusterDim.z = 1;
      cfg.attrs = attr;
      cfg.numAttrs = 1;
      int n_res;
      {
        std::lock_guard<std::mutex> lk(g_mu);
        if (st->resident[0][kk] == 0) {
          int n = 0;
          if (cudaOccupancyMaxActiveClusters(&n, kern_cluster, &cfg) != cudaSuccess) { (void)cudaGetLastError(); n = 0; }
          st->resident[0][kk] = n + 1;
        }
        n_res = st->resident[0][kk] - 1;
      }
      if ((long long)n_res * kk >= grid) {
        attn::FwdParams pc = p;
        pc.cluster_k = kk;
        pc.release_early = 1;
        if (launch_kernel(kern_cluster, grid, 512, smem, kk, stream, tq, tk, tv, to, pc) == cudaSuccess) {
          t_cluster_size = kk;
          return ATTN_OK;
        }
        (void)cudaGetLastError();                         // fall through to the plain launch
      }
    }
    if (!wait_roles_ok) return ATTN_ERR_BAD_TILES;        // (marker: the caller launches the last-finisher instantiation)
    ATTN_CUDA_TRY(launch_kernel(kern, grid, 512, smem, 0, stream, tq, tk, tv, to, p));
    return ATTN_OK;
  };
  bool fixed_roles = false;                              // of the instantiation that is launched
  const int ck = (t.tiles > 0 && t.ctas % t.tiles == 0) ? t.ctas / t.tiles : 0;
  const size_t c_landing = ck > 2 ? (size_t)((4 * NQ + ck - 1) / ck) * (ck - 1) * (32 * D * 4 + 256) : 0;
  if (p.causal && ck >= 2 && ck <= 4 && p.ratio >= 2 && c_landing <= (size_t)t.kv_stages * SM::kStageBytes) {
    // causal, ck CTAs per tile as one cluster: each a share of the tile's own key steps (the only way to run this grid)
    auto kern = attn::attn_fwd_kernel<D, TKV, NQ, true, true, true>;
    ATTN_ALLOW_SMEM(kern, smem);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(512);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = ck;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    attn::FwdParams pc = p;
    pc.cluster_k = ck;
    pc.release_early = 1;
    pc.seg_skip = -ck;
    // all clusters resident at once, else (or if the cluster launch fails) the same grid as equal ranges
    int n_res = 0;
    {
      std::lock_guard<std::mutex> lk(g_mu);
      if (st->resident[1][ck] == 0) {
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) { (void)cudaGetLastError(); n = 0; }
        st->resident[1][ck] = n + 1;
      }
      n_res = st->resident[1][ck] - 1;
    }
    if ((long long)n_res * ck >= grid && launch_kernel(kern, grid, 512, smem, ck, stream, tq, tk, tv, to, pc) == cudaSuccess) {
      t_cluster_size = ck;
      fixed_roles = true;
      rc = ATTN_OK;
    } else {
      (void)cudaGetLastError();
      rc = launch(attn::attn_fwd_kernel<D, TKV, NQ, true, false>);
    }
  } else if (p.causal) rc = launch(attn::attn_fwd_kernel<D, TKV, NQ, true, false>);
  else if (eager) {
    rc = launch_eager(attn::attn_fwd_kernel<D, TKV, NQ, false, true>, attn::attn_fwd_kernel<D, TKV, NQ, false, true, true>);
    fixed_roles = rc == ATTN_OK;
    if (rc == ATTN_ERR_BAD_TILES && !wait_roles_ok) rc = launch(attn::attn_fwd_kernel<D, TKV, NQ, false, false>);
  } else rc = launch(attn::attn_fwd_kernel<D, TKV, NQ, false, false>);
  if (rc != ATTN_OK) return rc;
  ATTN_CUDA_TRY(cudaGetLastError());
  t_launch_count = 1;
  launched(ATTN_KERNEL_TILED, grid, {"attn_fwd_kernel", 6, {D, TKV, NQ, p.causal, fixed_roles ? 1 : 0, t_cluster_size > 0 ? 1 : 0}});
  return ATTN_OK;
}

// Few query rows against many keys (decode_kernels.cuh).
template <int D, int MT, bool HALF>
int launch_decode(const void* q, const void* k, const void* v, void* o, int BH, int Lq, int Lk, int cluster_k, unsigned int* status,
                  int sms, cudaStream_t stream) {
  constexpr int kSlab = attn::decode_slab_keys(D);
  CUtensorMap tk, tv;
  int rc;
  if ((rc = make_tmap(&tk, k, BH, Lk, D, kSlab)) != ATTN_OK) return rc;
  if ((rc = make_tmap(&tv, v, BH, Lk, D, kSlab)) != ATTN_OK) return rc;
  attn::DecodeParams p;
  p.q = static_cast<const __nv_bfloat16*>(q);
  p.o = static_cast<__nv_bfloat16*>(o);
  p.Lq = Lq;
  p.Lk = Lk;
  p.cluster_k = cluster_k;
  p.scale_log2 = (float)(1.4426950408889634 / std::sqrt((double)D));
  p.status = status;
  // (launch_fwd says why.  Clusters of long CTAs that fill up to three quarters of the two places per SM, d = 64, 1 row, us early / when
  // the CTAs end: 24 x 16384 18.7 / 15.8, 96 x 4096 18.6 / 15.2; half as many keys a CTA 24 x 8192 9.7 / 10.2, more CTAs 64 x 4096 9.3 / 10.2)
  const long long ctas = (long long)BH * cluster_k;
  p.release_early = !(cluster_k > 1 && ctas > sms && 2 * ctas <= 3LL * sms && (long long)Lk * D * 4 / cluster_k >= 384 * 1024);
  auto kern = attn::attn_decode_kernel<D, MT, HALF>;
  constexpr int smem = attn::decode_smem_total<MT>();
  ATTN_ALLOW_SMEM(kern, smem);
  if (cluster_k > 8) ATTN_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  ATTN_CUDA_TRY(launch_kernel(kern, (long long)BH * cluster_k, 32 * attn::kDecodeWarps, smem, cluster_k, stream, tk, tv, p));
  t_cluster_size = cluster_k > 1 ? cluster_k : 0;
  t_launch_count = 1;
  launched(ATTN_KERNEL_FEW_ROWS, (long long)BH * cluster_k, {"attn_decode_kernel", 3, {D, MT, HALF ? 1 : 0}});
  return ATTN_OK;
}

// Clusters of k CTAs of the decode kernel that the device holds at once (0: none, or k CTAs are not allowed).
int resident_decode_clusters(int k) {
  auto kern = attn::attn_decode_kernel<128, 1, true>;
  constexpr int smem = attn::decode_smem_total<1>();
  int n = 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)k);
  cfg.blockDim = dim3(32 * attn::kDecodeWarps);
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = k;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess ||
      (k > 8 && cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) ||
      cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) {
    (void)cudaGetLastError();
    return 0;
  }
  return n;
}

// CTAs per head: a power of two (other cluster sizes leave SMs of a GPC unused).  Unit of the estimate: the time a CTA
// takes per slab when all slots are busy and HBM is the bound.  A CTA's start and end cost about 10 such units, k / 2 more
// for the cluster's barriers and merge; a partly full wave runs faster in proportion, down to 0.55, where a CTA with an SM to
// itself is bound by its own warps.  The slots are those the device reports for clusters of k: a cluster that has to wait for
// a second wave costs as much as a whole one.  Measured (us for k = 1 / 2 / 4 / 8): 256 heads x 4096 keys, d = 128:
// 83 / 81 / 87 / 101; 128 x 16384: 177 / 164 / 158 / 169; 32 x 4096: 39 / 22.5 / 15.0 / 15.2; 256 x 300: 9.2 / 14.5 / 21.4 /
// 39.5; k = 8 / 16: 8 x 16384: 24.2 / 18.0, 15 x 16384: 25.9 / 36.6.
int decode_split(int BH, int Lk, int d, const int (&clusters)[5]) {
  const int slabs = (Lk + attn::decode_slab_keys(d) - 1) / attn::decode_slab_keys(d);
  int best = 1;
  double best_cost = 0.0;
  for (int i = 0, k = 1; k <= attn::kDecodeMaxSplit; ++i, k *= 2) {
    if (k > 1 && (clusters[i] == 0 || slabs < attn::kDecodeWarps * k)) break;      // at least one slab per warp
    const double per_cta = (double)((slabs + k - 1) / k), ends = 10.0 + 0.5 * k;
    const double waves = (double)BH / std::max(1, clusters[i]), full = std::floor(waves), part = waves - full;
    const double cost = full * (per_cta + ends) + (part > 0.0 ? per_cta * std::max(part, 0.55) + ends : 0.0);
    if (k == 1 || cost < best_cost) { best = k; best_cost = cost; }
  }
  return best;
}

int dispatch_decode(const void* q, const void* k, const void* v, void* o, int BH, int Lq, int Lk, int d, unsigned int* status,
                    DeviceState* st, cudaStream_t s) {
  int clusters[5];
  {
    std::lock_guard<std::mutex> lk(g_mu);
    for (int i = 0; i < 5; ++i) {
      if (st->decode_clusters[i] == 0) st->decode_clusters[i] = resident_decode_clusters(1 << i) + 1;
      clusters[i] = st->decode_clusters[i] - 1;
    }
  }
  const int ck = decode_split(BH, Lk, d, clusters);
#define DECODE_CASE(D_)                                                                                          \
  if (d == D_) {                                                                                                 \
    if (Lq <= 8) return launch_decode<D_, 1, true>(q, k, v, o, BH, Lq, Lk, ck, status, st->desc.num_units, s);                       \
    if (Lq <= 16) return launch_decode<D_, 1, false>(q, k, v, o, BH, Lq, Lk, ck, status, st->desc.num_units, s);                     \
    return launch_decode<D_, 2, false>(q, k, v, o, BH, Lq, Lk, ck, status, st->desc.num_units, s);                                   \
  }
  DECODE_CASE(64)
  DECODE_CASE(128)
#undef DECODE_CASE
  return ATTN_ERR_UNSUPPORTED_SHAPE;
}

// Heads of a causal problem whose tiles are dealt out together, longest first: equal groups whose K and V take at most a third of the
// cache (32 heads of 8192, d = 128: 202 MB read from DRAM in groups of eight, 830 MB with 148 ranges that each walk a head of
// their own).  Equal, because a short last group would start its longest tiles when most CTAs have run dry.
int causal_group_heads(int BH, int L, int d, const attn_hw_desc& desc) {
  const long long at_most = std::max(1LL, desc.cache_bytes / (3 * 4LL * L * d));
  const long long groups = (BH + at_most - 1) / at_most;
  return (int)((BH + groups - 1) / groups);
}

// Whole Q tiles of 256 rows, one CTA each (pipe_kernel.cuh).  kernel_id: as what the launch is reported.
template <int D, bool CAUSAL>
int launch_pipe(const void* q, const void* k, const void* v, void* o, int BH, int Lq, int Lk, unsigned int* status, DeviceState* st,
                cudaStream_t stream, int kernel_id) {
  using SM = attn::PipeSmem<D>;
  CUtensorMap tq, tk, tv, to;
  int rc;
  if ((rc = make_tmap(&tq, q, BH, Lq, D, attn::kSub)) != ATTN_OK) return rc;
  if ((rc = make_tmap(&tk, k, BH, Lk, D, 128)) != ATTN_OK) return rc;
  if ((rc = make_tmap(&tv, v, BH, Lk, D, 128)) != ATTN_OK) return rc;
  if ((rc = make_tmap(&to, o, BH, Lq, D, 32)) != ATTN_OK) return rc;    // every warp stores its own 32 rows
  attn::PipeParams p;
  p.Lq = Lq;
  p.Lk = Lk;
  p.q_tiles = (Lq + 2 * attn::kSub - 1) / (2 * attn::kSub);
  p.n_steps = (Lk + 127) / 128;
  p.heads = BH;
  p.group_heads = causal_group_heads(BH, Lk, D, st->desc);
  p.stages = std::min(attn::kMaxStages, (st->desc.local_mem_bytes - SM::total(0)) / SM::kStageBytes) & ~1;
  p.scale_log2 = (float)(1.4426950408889634 / std::sqrt((double)D));
  p.status = status;
  const int smem = SM::total(p.stages);
  auto kern = attn::attn_pipe_kernel<D, CAUSAL>;
  ATTN_ALLOW_SMEM(kern, smem);
  ATTN_CUDA_TRY(launch_kernel(kern, (long long)BH * p.q_tiles, 512, smem, 0, stream, tq, tk, tv, to, p));
  t_cluster_size = 0;
  t_launch_count = 1;
  launched(kernel_id, (long long)BH * p.q_tiles, {"attn_pipe_kernel", 2, {D, CAUSAL ? 1 : 0}});
  return ATTN_OK;
}

// Whole Q tiles, one CTA each, a few softmax streams per tile (narrow_kernel.cuh).
template <int D, bool CAUSAL, int SUBS>
int launch_narrow(const void* q, const void* k, const void* v, void* o, int BH, int Lq, int Lk, unsigned int* status, DeviceState* st,
                  cudaStream_t stream) {
  using SM = attn::NarrowSmem<D, SUBS>;
  constexpr int kRings = attn::KvRings<SUBS>::kRings;
  CUtensorMap tq, tk, tv, to;
  int rc;
  if ((rc = make_tmap(&tq, q, BH, Lq, D, attn::kSub)) != ATTN_OK) return rc;
  if ((rc = make_tmap(&tk, k, BH, Lk, D, 128)) != ATTN_OK) return rc;
  if ((rc = make_tmap(&tv, v, BH, Lk, D, 128)) != ATTN_OK) return rc;
  if ((rc = make_tmap(&to, o, BH, Lq, D, 32)) != ATTN_OK) return rc;    // every warp stores its own 32 rows
  attn::NarrowParams p;
  p.Lq = Lq;
  p.Lk = Lk;
  p.q_tiles = (Lq + SUBS * attn::kSub - 1) / (SUBS * attn::kSub);
  p.n_steps = (Lk + 127) / 128;
  p.heads = BH;
  p.group_heads = causal_group_heads(BH, Lk, D, st->desc);
  p.stages = std::min(attn::kMaxStages, (st->desc.local_mem_bytes - SM::total(0)) / SM::kStageBytes) / kRings;
  p.scale_log2 = (float)(1.4426950408889634 / std::sqrt((double)D));
  p.status = status;
  const int smem = SM::total(kRings * p.stages);
  auto kern = attn::attn_narrow_kernel<D, CAUSAL, SUBS>;
  ATTN_ALLOW_SMEM(kern, smem);
  ATTN_CUDA_TRY(launch_kernel(kern, (long long)BH * p.q_tiles, attn::NarrowShape<D>::kThreads, smem, 0, stream, tq, tk, tv, to, p));
  t_cluster_size = 0;
  t_launch_count = 1;
  launched(CAUSAL ? ATTN_KERNEL_CAUSAL_TILES : ATTN_KERNEL_NARROW_TILES, (long long)BH * p.q_tiles,
           {"attn_narrow_kernel", 3, {D, CAUSAL ? 1 : 0, SUBS}});
  return ATTN_OK;
}

// Key steps of all heads of a causal problem in tiles of 256 rows.
long long causal_steps(int BH, int L) { return BH * attn_internal::head_units((L + 255) / 256, (L + 127) / 128, 2, 1); }

// Whether a causal plan of equal ranges runs as whole tiles instead.  Longest first, whole tiles take the longest tile's steps
// or an even share of all steps, one more per tile, whichever is more; 5 for the start and the end.  Measured (us in graphs, ranges /
// whole tiles): 128 heads x 4096, d = 128 571 / 471; 32 x 1111, d = 64 28.3 / 19.1; 16 x 4096, d = 128 89.6 / 72.4; where the longest
// tile decides, ranges stay: 8 x 4096 55.6 / (33 steps of 1.8) 61.4.  (Four ring stages: the MMA warps look that far ahead.)
bool causal_whole_tiles(const attn_tiles& t, int BH, int L, int d, int local_mem, int sms) {
  if (!t.causal || t.n_q != 2 || t.tile_kv != 128) return false;
  if (local_mem < (d == 64 ? attn::NarrowSmem<64, 2>::total(4) : attn::PipeSmem<128>::total(4))) return false;
  if (t.ctas % t.tiles == 0 && t.ctas > t.tiles) return false;      // clusters that share out each tile's own steps
  const long long even = (causal_steps(BH, L) + t.tiles + sms - 1) / sms;
  return std::max<long long>((L + 127) / 128, even) + 5 <= t.cost_steps;
}

// Sub-tiles a tile of narrow_kernel.cuh has: two, or one (tiles of 128 rows that take half as long), or 0 where another kernel
// stays.  Estimates in units of about 1.4 us at d = 64, in us at d = 128 (where a step of this kernel is slower than one of
// attn_fwd_kernel, 2.1 us against 1.75: its rows need every key tile for themselves).  Figures: us in graphs of 12 calls.
//   Causal.  One sub-tile where the longest tile would keep its CTA longer than an even share of the work, by the estimates
// (in steps) max(longest / 2, 1.1 even + 1) + 4.4 for one, max(longest, 1.1 even + 1) 0.96 + 4.1 for two and 1.08 times the plan's
// cost for its ranges (plan's kernel or two / one): 8 heads x 4096 40.8 / 30.9, 4 x 8192 61.4 / 52.1, 16 x 2048 29.9 / 19.8,
// 20 x 1111 18.6 / 12.6, 32 x 1111 19.1 / 16.4; on the other side 2 x 8192 41.8 / 50.9, 1 x 16384 62.6 / 95.9, 60 x 1500 37.5 / 39.8,
// 128 x 256 8.0 / 9.2.  A plan of clusters is launched as clusters, which attn_last_cluster_size reports and tests ask for, although one
// sub-tile is mostly faster there (9 x 1111 13.8 / 11.9, 16 x 512 10.2 / 8.0).
//   Not causal, one sub-tile: where 1.1 times the waves of half-length tiles and 2.8 are below the plan's cost (attn_fwd_kernel / one):
// 1 head x 256 7.2 / 5.5, 16 x 512 10.6 / 7.3, 16 x 1024 13.3 / 11.3, 32 x 1111 29.9 / 22.7, 60 x 1500 64.0 / 61.3; on the other
// side 128 x 256 7.9 / 8.4, 30 x 1024 17.2 / 19.1, 4 x 2048 15.5 / 17.6, 16 x 2048 28.8 / 32.3, 1 x 16384 95.4 / 98.3.  With more
// tiles than SMs the cost leaves out what a change of tile and a masked step take, and the kind of plan decides as well.  Whole tiles: only
// where half-length ones end in fewer than twice as many waves: 192 x 384 22.2 / 17.4, 111 x 512 19.3 / 16.0; as many 296 x 256
// 13.1 / 13.3, 96 x 1024 44.5 / 48.0, 85 x 1280 52.9 / 59.2; a single key step 256 x (512 x 128) 15.0 / 16.7, 61 x (3731 x 128) 24.4 /
// 26.8.  Tiles shared between CTAs, whose change and merge this kernel does not have: a masked last key tile 128 x 1000 71.0 / 60.9,
// 128 x 1300 116 / 113, few steps 222 x 640 51.9 / 47.5, few waves 48 x 1024 30.2 / 26.5; else 111 x 1536 98.0 / 104, 160 x 1280 105 / 109.
//   Not causal, two: whole waves of tiles, three or more with at most a tenth of all slots empty.  There a step of this kernel is
// 4 to 8 % slower than attn_fwd_kernel's until the power limit evens them out (attn_fwd_kernel / two: 148 x 1024 60.2 / 64.5, 74 x
// 2048 110 / 116, 148 x 4096 859 / 842, 128 x 8192 3009 / 2760), and a tile's end is cheaper: 48 key steps or more; shared tiles
// of up to 8 steps, 11 with a masked one (1000 x 256 50.7 / 39.3, 256 x 1000 128 / 114, 192 x 1300 172 / 154; 192 x 1280 126 / 131);
// whole tiles, four waves, up to 5 steps with a masked one, or a single step (296 x 450 41.0 / 38.9, 370 x (512 x 128) 18.8 / 17.6; three waves
// 444 x 256 17.7 / 17.6, 148 x 640 31.2 / 32.6).
//   The lines for calls that are not causal lie between this kernel and attn_fwd_kernel.  attn_pipe_kernel, which is asked after them, is
// faster than this one at some calls on this side: d = 64 128 x 1000 60.8 / 55.8, 256 x 1000 114 / 102, 192 x 1300 154 / 152, 296 x 450
// 39.1 / 36.5, d = 128 160 x 640 47.4 / 43.7.
//   d = 128, by the same reasoning.  Causal (plan's kernel or whole tiles / one): 8 heads x 4096 55.6 / 42.3, 16 x 2048 34.5 / 28.5, 20 x 1111
// 19.6 / 16.4, 1 x 256 8.9 / 7.3; on the other side 32 x 1111 20.3 / 22.9, 24 x 2048 33.3 / 39.3, 2 x 8192 51.0 / 71.5, 128 x 256
// 9.9 / 12.8.  (The estimates for the other kernels are of slower ones that were there before them.)  Not causal: 1 x 256 8.7 / 6.5, 16 x 512
// 12.3 / 9.6, 32 x 1111 36.5 / 30.0; on the other side 30 x 1024 19.8 / 23.4, 128 x 256 9.6 / 9.9, 16 x 2048 32.1 / 39.3, 1 x 16384
// 113 / 143.  Clusters stay here too (16 x 1024 15.9 / 14.3).
// A masked last key tile costs a tile of one sub-tile 2.4 us here (256 x 256 15.0, 256 x 200 23.9): with more tiles than SMs and whole
// ones only up to two waves (96 x 300 19.8 / 17.1; three 192 x 200 16.4 / 19.1, 96 x 450 23.4 / 25.9), and not beside two steps on more
// than half the SMs (48 x 130 8.7 / 8.9).  Else the waves may be half as many again as the plan's (192 x 384 26.1 / 21.8, 160 x 640 53.6 /
// 47.3; 111 x 768 44.4 / 45.6), whole tiles of up to three steps less than twice as many (370 x 256 22.2 / 19.8; 256 x 512 43.7 / 46.9),
// and a single step is not worth it (256 x (512 x 128) 21.2 / 23.2).
int narrow_subs(const attn_tiles& t, int BH, int Lq, int Lk, int d, int local_mem, int sms) {
  if (t.n_q != 2 || t.tile_kv != 128 || local_mem < (d == 64 ? attn::NarrowSmem<64, 2>::total(4) : attn::NarrowSmem<128, 1>::total(4))) return 0;
  const bool clusters = t.ctas % t.tiles == 0 && t.ctas > t.tiles;
  const long long half_tiles = (long long)BH * ((Lq + 127) / 128), steps = (Lk + 127) / 128;
  const long long waves = (half_tiles + sms - 1) / sms, plan_waves = (t.tiles + sms - 1) / sms;
  const bool shared = t.ctas < t.tiles, masked = Lk % 128 != 0;       // shared: one CTA per SM, tiles cut where its range ends
  if (d == 128) {
    if (clusters) return 0;
    if (!t.causal) {
      if (t.tiles <= sms ? masked && steps <= 2 && 2 * half_tiles > sms
          : steps < 2    ? true
          : masked && !shared ? waves > 2
                              : 2 * waves > 3 * plan_waves && (shared || steps > 3 || waves >= 2 * plan_waves))
        return 0;
      return 1.35 * (double)(waves * ((steps + 1) / 2)) + 2.3 < (double)t.cost_steps ? 1 : 0;
    }
    const double even = (double)causal_steps(BH, Lq) / sms;
    const double one = 5.5 + 2.1 * std::max(0.5 * (double)steps, 1.2 * even + 1.5);
    const double now = causal_whole_tiles(t, BH, Lq, d, local_mem, sms) ? 7.0 + 1.72 * std::max((double)steps, 1.1 * even + 1.0) : 1.7 * t.cost_steps;
    return one < now ? 1 : 0;
  }
  if (t.causal) {
    if (clusters) return 0;
    const double longest = (Lq + 127) / 128, share = 1.1 * (double)causal_steps(BH, Lq) / sms + 1.0;
    const double one = std::max(0.5 * longest, share) + 4.4;
    const bool whole = causal_whole_tiles(t, BH, Lq, d, local_mem, sms);
    const double now = whole ? 0.96 * std::max(longest, share) + 4.1 : 1.08 * t.cost_steps;
    return one < now ? 1 : whole ? 2 : 0;
  }
  if (t.tiles >= 3 * sms && 10 * plan_waves * sms <= 11LL * t.tiles) {
    const bool two = steps >= 48 || (shared ? steps <= (masked ? 11 : 8) : plan_waves >= 4 && (masked ? steps <= 5 : steps == 1));
    return two ? 2 : 0;
  }
  if (t.tiles > sms && (steps < 2 || (shared ? !masked && steps > 6 && (waves > 4 || steps > 12) : waves >= 2 * plan_waves))) return 0;
  return 1.1 * (double)(waves * ((steps + 1) / 2)) + 2.8 < (double)t.cost_steps ? 1 : 0;
}

// Calls, not causal, that pipe_kernel.cuh takes over from attn_fwd_kernel, at either head dimension (us in graphs of 8 to 40 calls, attn_fwd_kernel / this).
//   Plans of whole tiles, d = 128: with more tiles than SMs always (95 shapes, 0.91 times on the geometric mean: 592 x 512 75.8 / 63.2).  One wave: from four
// key steps on (three and fewer 0.98 to 1.05) where the tiles fill three quarters of the SMs (128 x (256 x 1000) 0.97 times; 104 x (256 x
// 1280) 22.6 / 24.8, 10 x 2560 38.7 / 39.7).  From a dozen steps on without a masked one this kernel is 1 to 2 % slower in a burst of some
// milliseconds and as much faster in a loop of seconds, under the power limit (8 x 4096 66.5 / 65.9, 74 x (1000 x 2048) 79.5 / 78.9, 37 x (4096 x 2560)
// 185 / 182): the line is drawn for loops.
//   d = 64: its step takes one cubic and two quartics of eight pairs where attn_fwd_kernel takes two cubics, which costs 2 % of a step and leaves
// long tiles to that kernel.  One wave from 4 key steps (3: 64 x 384 10.0 / 10.2) to 10 (148 x (256 x 1280) 20.7 / 20.2; 20 x (1700 x 1700)
// 25.7 / 26.3); two waves to 17, three to 23, four to 29 (32 x 2048 54.0 / 53.5, 32 x 2304 59.4 / 60.2, 24 x 3000 77.6 / 78.9, 37 x 4000
// 205 / 208), more to 31, where the last wave is full to 23 (60 x 3000 203 / 195, 111 x 3000 352 / 352, 74 x 4096 408 / 414).  A head whose last
// tile has only one sub-tile gains nothing there: the sub-tile takes nearly as long alone.  In full waves of whole tiles such calls stay from 3 steps on, with a
// masked one, which attn_fwd_kernel is slow at, from 12 (148 x 640 31.2 / 32.8, 148 x (1100 x 512) 1.056 times, 148 x 1111 1.00; 148 x (1280 x 512) 0.945).  Of 554
// shapes on two grids 442 go here, 0.959 times, six of them slower by 1 to 2.7 %.
//   Plans whose tiles are cut over the machine: where whole tiles are estimated to be faster by 2 % (d = 64) or 4 %.  The estimates are
// fits in us, of this kernel over its waves and key steps and of the plan's over its cost, that miss by 4 to 7 % (one sd): of 140 shapes
// 49 go here, 0.89 times on the geometric mean and none slower by more than 1 %; 14 that would be 3 % faster or more stay.
bool pipe_tiles(const attn_tiles& t, int Lq, int Lk, int d, int local_mem, int sms) {
  if (t.causal || t.n_q != 2 || t.tile_kv != 128) return false;
  if (local_mem < (d == 64 ? attn::PipeSmem<64>::total(4) : attn::PipeSmem<128>::total(4))) return false;
  const int steps = (Lk + 127) / 128, waves = (t.tiles + sms - 1) / sms;
  const long long filled = 100LL * t.tiles / ((long long)waves * sms);       // per cent of the waves' slots
  if (waves == 1) return t.ctas == t.tiles && steps >= 4 && (d == 64 ? steps <= 10 : 4 * t.tiles >= 3 * sms);
  if (d == 64) {
    if (steps >= 32 || steps >= 6 + 6 * waves || (filled >= 98 && steps >= 24)) return false;
    if (t.ctas == t.tiles && filled >= 97 && (Lq - 1) % 256 < 128 && steps >= (Lk % 128 ? 12 : 3)) return false;
  }
  if (t.ctas == t.tiles) return true;
  if (t.ctas > t.tiles) return false;
  const double whole = d == 64 ? 3.0 + waves * (2.0 + 1.376 * steps + (Lk % 128 ? 0.35 : 0.0)) : 4.0 + waves * (2.3 + 1.647 * steps);
  const double cut = d == 64 ? 2.5 + 1.493 * t.cost_steps : 5.7 + 1.78 * t.cost_steps;
  return whole < (d == 64 ? 0.98 : 0.96) * cut;
}

int dispatch_fwd(const void* q, const void* k, const void* v, void* o, int B, int H, int L, int d,
                 const attn_tiles& t, float* ws, unsigned int* status, DeviceState* st, cudaStream_t s, int Lk = 0,
                 bool may_overlap = false, bool own_plan = false) {
  if (Lk == 0) Lk = L;
  // own_plan: the device's own, with no field changed and from no caller's descriptor -- those say how many CTAs run
  const int sms = st->desc.num_units;
  if (own_plan) {
    if (const int subs = narrow_subs(t, B * H, L, Lk, d, st->desc.local_mem_bytes, sms)) {
      auto launch = d == 128 ? (t.causal ? launch_narrow<128, true, 1> : launch_narrow<128, false, 1>)
                    : t.causal ? (subs == 1 ? launch_narrow<64, true, 1> : launch_narrow<64, true, 2>)
                               : (subs == 1 ? launch_narrow<64, false, 1> : launch_narrow<64, false, 2>);
      return launch(q, k, v, o, B * H, L, Lk, status, st, s);
    }
    if (d == 128 && Lk == L && causal_whole_tiles(t, B * H, L, d, st->desc.local_mem_bytes, sms))
      return launch_pipe<128, true>(q, k, v, o, B * H, L, L, status, st, s, ATTN_KERNEL_CAUSAL_TILES);
    if (pipe_tiles(t, L, Lk, d, st->desc.local_mem_bytes, sms))
      return d == 64 ? launch_pipe<64, false>(q, k, v, o, B * H, L, Lk, status, st, s, ATTN_KERNEL_TILED)
                     : launch_pipe<128, false>(q, k, v, o, B * H, L, Lk, status, st, s, ATTN_KERNEL_TILED);
  }
#define ATTN_CASE(D_, TKV_, NQ_) \
  if (d == D_ && t.tile_kv == TKV_ && t.n_q == NQ_) \
    return launch_fwd<D_, TKV_, NQ_>(q, k, v, o, B, H, L, Lk, t, ws, status, st, s, may_overlap);
  ATTN_CASE(128, 128, 2)
  ATTN_CASE(128, 64, 2)
  ATTN_CASE(128, 128, 1)
  ATTN_CASE(128, 64, 1)
  ATTN_CASE(64, 128, 2)
  ATTN_CASE(64, 64, 2)
  ATTN_CASE(64, 128, 1)
  ATTN_CASE(64, 64, 1)
#undef ATTN_CASE
  return ATTN_ERR_BAD_TILES;
}

// Calls that the decode kernel takes over from the tiled one.  Up to 16 rows (at d = 64 up to 32) it is as fast or faster at every
// size measured (1.0-5 times).  17 to 32 rows at d = 128 keep its warps as busy as HBM: there only where the tiled kernel would
// run whole tiles in waves and leave an eighth of their slots empty, in an even number of waves (two of them are one of the
// decode kernel's, which has two CTAs per SM), over 750 keys a wave or more (us tiled / decode, 24 rows: 192 heads x 2048 keys
// 55.7 / 49.6, 256 x 4096 103 / 88; 32 rows: 256 x 1500 48.5 / 44.5, 500 x 3000 158 / 140).  On the other side, 32 rows:
// 256 x 1280 39.8 / 40.0, 296 x 4096 103 / 110, 350 x 1280 57 / 74, 444 x 1024 48 / 65.
bool decode_rows(int Lq, int Lk, int d, const attn_tiles& t, int sms) {
  if (Lq <= 16 || (d == 64 && Lq <= 32)) return true;
  const long long waves = (t.tiles + sms - 1) / sms;
  return Lq <= 32 && t.ctas == t.tiles && waves % 2 == 0 && 8LL * t.tiles <= 7LL * waves * sms && Lk >= 750LL * waves;
}

// A plan needs the workspace unless every CTA owns exactly one whole Q tile.
bool plan_needs_workspace(const attn_tiles& t) { return t.causal != 0 || t.ctas != t.tiles; }

// A workspace handed to one call (attn_forward_ws) instead of the one registered for the device.
struct CallWorkspace {
  void* ws;
  size_t bytes;
  unsigned int* status;
};

int forward_impl(const void* q, const void* k, const void* v, void* o, int B, int H, int L, int d, int causal,
                 const attn_tiles* ovr, void* cuda_stream, const attn_hw_desc* plan_desc = nullptr, int Lk = 0,
                 const CallWorkspace* call_ws = nullptr) {
  t_launch_count = 0;
  if (Lk == 0) Lk = L;                       // keys per head; L is the number of query rows per head
  int rc = check_args(q, k, v, o, B, H, L, d, Lk);
  if (rc != ATTN_OK) return rc;
  if (Lk != L && (causal || (ovr && ovr->causal))) return ATTN_ERR_UNSUPPORTED_SHAPE;
  DeviceState* st = nullptr;
  if ((rc = device_state(&st)) != ATTN_OK) return rc;
  if (ovr && ovr->causal) causal = 1;
  if (plan_desc) {
    // a caller-supplied descriptor must describe this device or a smaller machine of the same architecture
    const attn_hw_desc& a = *plan_desc;
    const attn_hw_desc& dv = st->desc;
    if (a.struct_bytes != (int32_t)sizeof(attn_hw_desc)) return ATTN_ERR_INVALID_ARG;
    if (a.num_units < 1 || a.num_units > dv.num_units || a.local_mem_bytes > dv.local_mem_bytes ||
        a.regs_per_unit > dv.regs_per_unit || a.acc_mem_columns > dv.acc_mem_columns || a.acc_mem_columns <= 0 ||
        a.acc_mem_lanes != dv.acc_mem_lanes || a.atom_m != dv.atom_m || a.atom_n != dv.atom_n || a.atom_k != dv.atom_k ||
        a.atom_n_max > dv.atom_n_max || a.elem_bytes != dv.elem_bytes || a.simd_width != dv.simd_width)
      return ATTN_ERR_INVALID_ARG;
  }
  const attn_hw_desc& desc = plan_desc ? *plan_desc : st->desc;
  attn_tiles t;
  if ((rc = attn_internal::plan_qk(&desc, B, H, L, Lk, d, causal, &t)) != ATTN_OK) return rc;
  if (!t.feasible) return ATTN_ERR_INFEASIBLE_PLAN;
  if (ovr) {
    if (ovr->n_q > 0) t.n_q = ovr->n_q;
    if (ovr->tile_kv > 0) t.tile_kv = ovr->tile_kv;
    if (t.n_q != 1 && t.n_q != 2) return ATTN_ERR_BAD_TILES;
    if (t.tile_kv != 64 && t.tile_kv != 128) return ATTN_ERR_BAD_TILES;
    const int q_bytes = t.n_q * 128 * d * 2, stage = t.tile_kv * d * 2;
    const int reserve = 3072 + t.n_q * 128 * 128;   // barriers etc. + output staging (see FwdSmem)
    int max_stages = (desc.local_mem_bytes - q_bytes - reserve) / stage;
    if (max_stages > attn::kMaxStages) max_stages = attn::kMaxStages;
    t.kv_stages = ovr->kv_stages > 0 ? ovr->kv_stages : max_stages;
    if (t.kv_stages < 2 || t.kv_stages > max_stages) return ATTN_ERR_BAD_TILES;
    t.tile_q = t.n_q * 128;
    t.tiles = B * H * ((L + t.tile_q - 1) / t.tile_q);
    // grid: ctas if given, else kv_splits CTAs per Q tile if given, else the planner's occupancy rule
    // re-applied to the overridden tile shape
    const int steps = (Lk + t.tile_kv - 1) / t.tile_kv;
    if (ovr->ctas > 0) {
      t.ctas = ovr->ctas;
    } else if (ovr->kv_splits > 0) {
      t.ctas = t.tiles * ovr->kv_splits;
    } else {
      t.ctas = attn_internal::grid_size(desc, B * H, (L + t.tile_q - 1) / t.tile_q, steps, t.tile_q / t.tile_kv, causal,
                                        2LL * Lk * d * desc.elem_bytes, 4 * t.n_q, d, (long long)t.kv_stages * stage).ctas;
    }
    t.kv_splits = (t.ctas + t.tiles - 1) / t.tiles;
    if (t.ctas < 1) return ATTN_ERR_BAD_TILES;
    t.smem_bytes = q_bytes + t.kv_stages * stage + reserve;
  }
  float* ws = nullptr;
  if (plan_needs_workspace(t)) {
    const size_t need = attn_workspace_bytes(&t, B, H, L, d);
    if (call_ws) {
      if (!call_ws->ws || call_ws->bytes < need) return ATTN_ERR_NEED_WORKSPACE;
      ws = static_cast<float*>(call_ws->ws);
    } else {
      std::lock_guard<std::mutex> lk(g_mu);
      if (!st->ws || st->ws_bytes < need) return ATTN_ERR_NEED_WORKSPACE;
      ws = static_cast<float*>(st->ws);
    }
  }
  if (!ovr && !plan_desc && !call_ws && Lk != L && decode_rows(L, Lk, d, t, st->desc.num_units))
    return dispatch_decode(q, k, v, o, B * H, L, Lk, d, nullptr, st, static_cast<cudaStream_t>(cuda_stream));
  return dispatch_fwd(q, k, v, o, B, H, L, d, t, ws, call_ws ? call_ws->status : nullptr, st,
                      static_cast<cudaStream_t>(cuda_stream), Lk, call_ws != nullptr, !ovr && !plan_desc);
}

template <int D, int TKV>
int launch_simple(const void* q, const void* k, const void* v, void* o, int B, int H, int L, float* scores_out,
                  cudaStream_t stream) {
  const int BH = B * H;
  CUtensorMap tq, tk, tv;
  int rc;
  if ((rc = make_tmap(&tq, q, BH, L, D, attn::kSub)) != ATTN_OK) return rc;
  if ((rc = make_tmap(&tk, k, BH, L, D, TKV)) != ATTN_OK) return rc;
  if ((rc = make_tmap(&tv, v, BH, L, D, TKV)) != ATTN_OK) return rc;
  const int smem = attn::kSub * D * 2 + 2 * TKV * D * 2 + 1024;
  auto kern = attn::attn_fwd_simple_kernel<D, TKV>;
  ATTN_ALLOW_SMEM(kern, smem);
  const float scale_log2 = (float)(1.4426950408889634 / std::sqrt((double)D));
  dim3 grid((L + attn::kSub - 1) / attn::kSub, BH);
  kern<<<grid, 128, smem, stream>>>(tq, tk, tv, reinterpret_cast<__nv_bfloat16*>(o), L, scale_log2, scores_out);
  ATTN_CUDA_TRY(cudaGetLastError());
  t_launch_count = 1;
  launched(ATTN_KERNEL_SIMPLE, (long long)grid.x * grid.y, {"attn_fwd_simple_kernel", 2, {D, TKV}});
  return ATTN_OK;
}

}  // namespace

extern "C" int attn_hw_desc_query(int device, attn_hw_desc* out) {
  if (!out) return ATTN_ERR_INVALID_ARG;
  int major = 0, minor = 0, sms = 0, smem_optin = 0, regs = 0, clock_khz = 0;
  ATTN_CUDA_TRY(cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, device));
  ATTN_CUDA_TRY(cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, device));
  if (major != 10) return ATTN_ERR_WRONG_ARCH;
  attn_hw_desc_b200(out);  // per-architecture constants (tensor memory, atom shapes)
  ATTN_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device));
  ATTN_CUDA_TRY(cudaDeviceGetAttribute(&smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device));
  ATTN_CUDA_TRY(cudaDeviceGetAttribute(&regs, cudaDevAttrMaxRegistersPerMultiprocessor, device));
  int l2 = 0;
  ATTN_CUDA_TRY(cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, device));
  if (l2 > 0) out->cache_bytes = l2;
  ATTN_CUDA_TRY(cudaDeviceGetAttribute(&clock_khz, cudaDevAttrClockRate, device));
  out->num_units = sms;
  out->local_mem_bytes = smem_optin;
  out->regs_per_unit = regs;
  // dense bf16: 8192 FLOP per clock per SM at the device's maximum SM clock
  out->peak_tflops = 8192.0 * sms * (clock_khz * 1e3) / 1e12;
  // Resident clusters of k CTAs, asked for the kernel that uses them at its largest shared-memory footprint.
  {
    int cur = 0;
    ATTN_CUDA_TRY(cudaGetDevice(&cur));
    if (cur != device) ATTN_CUDA_TRY(cudaSetDevice(device));
    auto kern = attn::attn_fwd_kernel<128, 128, 2, false, true, true>;
    const int smem = attn::FwdSmem<128, 128, 2>::total(4);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    for (int k = 1; k <= 8; ++k) {
      int n = 0;
      if (e == cudaSuccess) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)(sms / k * k));
        cfg.blockDim = dim3(512);
        cfg.dynamicSmemBytes = smem;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = k;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) n = 0;
      }
      out->max_clusters[k - 1] = n;
    }
    (void)cudaGetLastError();
    if (cur != device) ATTN_CUDA_TRY(cudaSetDevice(cur));
  }
  return ATTN_OK;
}

extern "C" int attn_set_workspace(int device, void* dev_ptr, size_t bytes) {
  if (device < 0 || device >= kMaxDevices) return ATTN_ERR_INVALID_ARG;
  if (dev_ptr && ((uintptr_t)dev_ptr & 15u)) return ATTN_ERR_MISALIGNED;
  if (dev_ptr && bytes >= (size_t)attn::kCounterBytes) {
    // arrival counters at the head of the workspace start at zero; kernels leave them at zero
    ATTN_CUDA_TRY(cudaMemset(dev_ptr, 0, attn::kCounterBytes));
  }
  std::lock_guard<std::mutex> lk(g_mu);
  g_dev[device].ws = dev_ptr;
  g_dev[device].ws_bytes = dev_ptr ? bytes : 0;
  return ATTN_OK;
}

extern "C" int attn_forward(const void* q, const void* k, const void* v, void* o, int B, int H, int L, int d,
                            void* cuda_stream) {
  return forward_impl(q, k, v, o, B, H, L, d, 0, nullptr, cuda_stream);
}

extern "C" int attn_workspace_init(void* workspace, size_t workspace_bytes, uint32_t* status_dev, void* cuda_stream) {
  if (!workspace && !status_dev) return ATTN_ERR_INVALID_ARG;
  if (workspace && (((uintptr_t)workspace & 15u) || workspace_bytes < (size_t)attn::kCounterBytes)) return ATTN_ERR_INVALID_ARG;
  if (status_dev && ((uintptr_t)status_dev & 15u)) return ATTN_ERR_MISALIGNED;
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  if (workspace) ATTN_CUDA_TRY(cudaMemsetAsync(workspace, 0, attn::kCounterBytes, s));
  if (status_dev) ATTN_CUDA_TRY(cudaMemsetAsync(status_dev, 0, 4 * sizeof(uint32_t), s));
  return ATTN_OK;
}

extern "C" int attn_forward_ws(const void* q, const void* k, const void* v, void* o, int B, int H, int L, int d, int causal,
                               void* workspace, size_t workspace_bytes, uint32_t* status_dev, void* cuda_stream) {
  if (workspace && ((uintptr_t)workspace & 15u)) return ATTN_ERR_MISALIGNED;
  if (status_dev && ((uintptr_t)status_dev & 15u)) return ATTN_ERR_MISALIGNED;
  const CallWorkspace cw = {workspace, workspace ? workspace_bytes : 0, status_dev};
  return forward_impl(q, k, v, o, B, H, L, d, causal ? 1 : 0, nullptr, cuda_stream, nullptr, 0, &cw);
}

extern "C" int attn_status_read(uint32_t* status_dev, void* workspace, void* cuda_stream, uint32_t* detail) {
  if (!status_dev) return ATTN_ERR_INVALID_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  ATTN_CUDA_TRY(cudaStreamSynchronize(s));
  unsigned int h[4] = {0, 0, 0, 0};
  ATTN_CUDA_TRY(cudaMemcpy(h, status_dev, sizeof h, cudaMemcpyDeviceToHost));
  if (detail)
    for (int i = 0; i < 4; ++i) detail[i] = h[i];
  if (h[0] == 0) return ATTN_OK;
  // the aborted launch may have left arrival counters non-zero
  ATTN_CUDA_TRY(cudaMemset(status_dev, 0, sizeof h));
  if (workspace) ATTN_CUDA_TRY(cudaMemset(workspace, 0, attn::kCounterBytes));
  return ATTN_ERR_DEVICE_TIMEOUT;
}

extern "C" int attn_forward_qk(const void* q, const void* k, const void* v, void* o, int B, int H, int Lq, int Lk, int d,
                               void* cuda_stream) {
  if (Lk <= 0) return ATTN_ERR_INVALID_ARG;
  return forward_impl(q, k, v, o, B, H, Lq, d, 0, nullptr, cuda_stream, nullptr, Lk);
}

extern "C" int attn_forward_causal(const void* q, const void* k, const void* v, void* o, int B, int H, int L, int d,
                                   void* cuda_stream) {
  return forward_impl(q, k, v, o, B, H, L, d, 1, nullptr, cuda_stream);
}

extern "C" int attn_forward_call(const attn_call* c) {
  if (!c || c->Lk <= 0) return ATTN_ERR_INVALID_ARG;
  return forward_impl(c->q, c->k, c->v, c->o, c->B, c->H, c->Lq, c->d, c->causal ? 1 : 0, nullptr, c->cuda_stream, nullptr, c->Lk);
}

extern "C" int attn_forward_desc(const attn_hw_desc* desc, const void* q, const void* k, const void* v, void* o, int B, int H,
                                 int L, int d, int causal, void* cuda_stream) {
  if (!desc) return ATTN_ERR_INVALID_ARG;
  return forward_impl(q, k, v, o, B, H, L, d, causal ? 1 : 0, nullptr, cuda_stream, desc);
}

extern "C" int attn_forward_tiles(const void* q, const void* k, const void* v, void* o, int B, int H, int L, int d,
                                  const attn_tiles* override_tiles, void* cuda_stream) {
  return forward_impl(q, k, v, o, B, H, L, d, 0, override_tiles, cuda_stream);
}

extern "C" int attn_forward_simple(const void* q, const void* k, const void* v, void* o, int B, int H, int L, int d,
                                   int tile_kv, float* scores_out, void* cuda_stream) {
  t_launch_count = 0;
  int rc = check_args(q, k, v, o, B, H, L, d);
  if (rc != ATTN_OK) return rc;
  DeviceState* st = nullptr;
  if ((rc = device_state(&st)) != ATTN_OK) return rc;
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  if (d == 128 && tile_kv == 128) return launch_simple<128, 128>(q, k, v, o, B, H, L, scores_out, s);
  if (d == 128 && tile_kv == 64) return launch_simple<128, 64>(q, k, v, o, B, H, L, scores_out, s);
  if (d == 64 && tile_kv == 128) return launch_simple<64, 128>(q, k, v, o, B, H, L, scores_out, s);
  if (d == 64 && tile_kv == 64) return launch_simple<64, 64>(q, k, v, o, B, H, L, scores_out, s);
  return ATTN_ERR_BAD_TILES;
}

namespace {
// Streams and events of the host-buffer entry point's copy/compute pipeline, created on first use per device.
constexpr int kHostBlocksMax = 2;
struct HostPipe {
  cudaStream_t in = nullptr, out = nullptr;
  cudaEvent_t start = nullptr, done = nullptr, loaded[kHostBlocksMax] = {}, computed[kHostBlocksMax] = {};
  bool ok = false;
};
HostPipe g_pipe[kMaxDevices];
std::mutex g_pipe_mu;

HostPipe* host_pipe() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return nullptr;
  HostPipe& hp = g_pipe[dev];
  if (!hp.ok) {
    bool good = cudaStreamCreateWithFlags(&hp.in, cudaStreamNonBlocking) == cudaSuccess &&
                cudaStreamCreateWithFlags(&hp.out, cudaStreamNonBlocking) == cudaSuccess &&
                cudaEventCreateWithFlags(&hp.start, cudaEventDisableTiming) == cudaSuccess &&
                cudaEventCreateWithFlags(&hp.done, cudaEventDisableTiming) == cudaSuccess;
    for (int i = 0; good && i < kHostBlocksMax; ++i)
      good = cudaEventCreateWithFlags(&hp.loaded[i], cudaEventDisableTiming) == cudaSuccess &&
             cudaEventCreateWithFlags(&hp.computed[i], cudaEventDisableTiming) == cudaSuccess;
    if (!good) { (void)cudaGetLastError(); return nullptr; }
    hp.ok = true;
  }
  return &hp;
}

// The blocks of query rows of the pipelined host path (one long head): kHostBlocksMax blocks of at least 4096
// rows, a multiple of 256 each but the last.  Returns the number of blocks, 0 if not pipelined.
// (Measured at L = 16384, d = 128: unsplit 0.450 ms, two blocks 0.398 ms, four blocks 0.475 ms -- a 4096-row
// launch against 16384 keys fills the machine worse than the copies it hides.)
int host_split(int B, int H, int L, int rows[kHostBlocksMax]) {
  if ((long long)B * H != 1 || L < 8192) return 0;
  const int n = std::min(kHostBlocksMax, L / 4096);
  const int per = ((L + n - 1) / n + 255) / 256 * 256;
  int left = L, c = 0;
  for (; c < n && left > 0; ++c) { rows[c] = std::min(per, left); left -= rows[c]; }
  return c;
}
}  // namespace

extern "C" size_t attn_forward_host_workspace_bytes(const attn_hw_desc* desc, int B, int H, int L, int d) {
  attn_tiles t;
  if (!desc || attn_plan(desc, B, H, L, d, &t) != ATTN_OK || !t.feasible) return 0;
  size_t need = attn_workspace_bytes(&t, B, H, L, d);
  int rows[kHostBlocksMax];
  const int blocks = host_split(B, H, L, rows);
  for (int c = 0; c < blocks; ++c)
    if (c == 0 || rows[c] != rows[c - 1])
      if (attn_plan_qk(desc, B, H, rows[c], L, d, &t) == ATTN_OK && t.feasible)
        need = std::max(need, attn_workspace_bytes(&t, B, H, rows[c], d));
  return need;
}

extern "C" int attn_forward_host(const void* q_host, const void* k_host, const void* v_host, void* o_host, int B,
                                 int H, int L, int d, void* dev_scratch, size_t dev_scratch_bytes,
                                 void* cuda_stream) {
  if (!q_host || !k_host || !v_host || !o_host || !dev_scratch || B <= 0 || H <= 0 || L <= 0 || d <= 0)
    return ATTN_ERR_INVALID_ARG;
  const size_t bytes = (size_t)B * H * L * d * 2;
  if (dev_scratch_bytes < 4 * bytes || ((uintptr_t)dev_scratch & 255u)) return ATTN_ERR_INVALID_ARG;
  char* base = static_cast<char*>(dev_scratch);
  char *dq = base, *dk = base + bytes, *dv = base + 2 * bytes, *dout = base + 3 * bytes;
  int rc = check_args(dq, dk, dv, dout, B, H, L, d);
  if (rc != ATTN_OK) return rc;
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  // One long head: the query rows go in blocks (every query row attends to all keys, so the blocks are
  // independent problems of attn_forward_qk).  K, V and the first block are copied, then each later block's copy
  // runs under the kernel before it and each block's result leaves under the kernel after it.
  // The copies use two streams of the library's own; the caller's stream sees the call as one unit of work.
  int rows[kHostBlocksMax];
  const int blocks = host_split(B, H, L, rows);
  if (blocks > 0) {
    std::lock_guard<std::mutex> lk(g_pipe_mu);
    HostPipe* hp = host_pipe();
    if (hp) {
      int first[kHostBlocksMax] = {};
      for (int c = 1; c < blocks; ++c) first[c] = first[c - 1] + rows[c - 1];
      const char *qh = static_cast<const char*>(q_host);
      char* oh = static_cast<char*>(o_host);
      const size_t row_bytes = (size_t)d * 2;
      ATTN_CUDA_TRY(cudaEventRecord(hp->start, s));
      ATTN_CUDA_TRY(cudaStreamWaitEvent(hp->in, hp->start, 0));
      ATTN_CUDA_TRY(cudaMemcpyAsync(dk, k_host, bytes, cudaMemcpyHostToDevice, hp->in));
      ATTN_CUDA_TRY(cudaMemcpyAsync(dv, v_host, bytes, cudaMemcpyHostToDevice, hp->in));
      for (int c = 0; c < blocks; ++c) {
        ATTN_CUDA_TRY(cudaMemcpyAsync(dq + first[c] * row_bytes, qh + first[c] * row_bytes, rows[c] * row_bytes,
                                      cudaMemcpyHostToDevice, hp->in));
        ATTN_CUDA_TRY(cudaEventRecord(hp->loaded[c], hp->in));
      }
      int launches = 0;
      for (int c = 0; c < blocks; ++c) {
        ATTN_CUDA_TRY(cudaStreamWaitEvent(s, hp->loaded[c], 0));
        rc = forward_impl(dq + first[c] * row_bytes, dk, dv, dout + first[c] * row_bytes, 1, 1, rows[c], d, 0, nullptr,
                          cuda_stream, nullptr, L);
        if (rc != ATTN_OK) break;
        launches += t_launch_count;
        ATTN_CUDA_TRY(cudaEventRecord(hp->computed[c], s));
        ATTN_CUDA_TRY(cudaStreamWaitEvent(hp->out, hp->computed[c], 0));
        ATTN_CUDA_TRY(cudaMemcpyAsync(oh + first[c] * row_bytes, dout + first[c] * row_bytes, rows[c] * row_bytes,
                                      cudaMemcpyDeviceToHost, hp->out));
      }
      // the caller's stream continues only after every copy of this call
      ATTN_CUDA_TRY(cudaEventRecord(hp->done, hp->out));
      ATTN_CUDA_TRY(cudaStreamWaitEvent(s, hp->done, 0));
      ATTN_CUDA_TRY(cudaStreamWaitEvent(s, hp->loaded[blocks - 1], 0));
      t_launch_count = launches;
      return rc;
    }
  }
  ATTN_CUDA_TRY(cudaMemcpyAsync(dq, q_host, bytes, cudaMemcpyHostToDevice, s));
  ATTN_CUDA_TRY(cudaMemcpyAsync(dk, k_host, bytes, cudaMemcpyHostToDevice, s));
  ATTN_CUDA_TRY(cudaMemcpyAsync(dv, v_host, bytes, cudaMemcpyHostToDevice, s));
  rc = forward_impl(dq, dk, dv, dout, B, H, L, d, 0, nullptr, cuda_stream);
  if (rc != ATTN_OK) return rc;
  ATTN_CUDA_TRY(cudaMemcpyAsync(o_host, dout, bytes, cudaMemcpyDeviceToHost, s));
  return ATTN_OK;
}

// ---------------------------------------------------------------------------------------------
// Allocation-free entry point.  The scratch that a split plan needs (arrival counters followed by
// the partial outputs) is this file-scope device array instead of a caller-supplied workspace.
// In host code the name below is only a handle: its device address is obtained once per device
// with cudaGetSymbolAddress and that pointer is what the kernel receives.
// ---------------------------------------------------------------------------------------------
static __device__ __align__(256) unsigned char g_attn_static_scratch[ATTN_STATIC_SCRATCH_BYTES];

namespace {
void* g_static_scratch_ptr[kMaxDevices] = {};
std::mutex g_static_mu;

// Device address of the array on the current device, looked up on first use.
int static_scratch_address(void** out) {
  int dev = 0;
  ATTN_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) return ATTN_ERR_INVALID_ARG;
  std::lock_guard<std::mutex> lk(g_static_mu);
  if (!g_static_scratch_ptr[dev]) {
    void* ptr = nullptr;
    ATTN_CUDA_TRY(cudaGetSymbolAddress(&ptr, g_attn_static_scratch));
    if (!ptr) return ATTN_ERR_CUDA;
    g_static_scratch_ptr[dev] = ptr;
  }
  *out = g_static_scratch_ptr[dev];
  return ATTN_OK;
}
}  // namespace

extern "C" int attn_forward_static_scratch(const void* q, const void* k, const void* v, void* o, int B, int H, int L,
                                           int d, void* cuda_stream) {
  t_launch_count = 0;
  int rc = check_args(q, k, v, o, B, H, L, d);
  if (rc != ATTN_OK) return rc;
  DeviceState* st = nullptr;
  if ((rc = device_state(&st)) != ATTN_OK) return rc;
  attn_tiles t;
  if ((rc = attn_plan(&st->desc, B, H, L, d, &t)) != ATTN_OK) return rc;
  if (!t.feasible) return ATTN_ERR_INFEASIBLE_PLAN;
  void* scratch = nullptr;
  if ((rc = static_scratch_address(&scratch)) != ATTN_OK) return rc;
  cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
  if (plan_needs_workspace(t)) {
    if (attn_workspace_bytes(&t, B, H, L, d) > (size_t)ATTN_STATIC_SCRATCH_BYTES) return ATTN_ERR_SCRATCH_LIMIT;
    // the array keeps the previous call's contents: the arrival counters must start at zero
    ATTN_CUDA_TRY(cudaMemsetAsync(scratch, 0, attn::kCounterBytes, stream));
  }
  return dispatch_fwd(q, k, v, o, B, H, L, d, t, static_cast<float*>(scratch), nullptr, st, stream);
}

namespace {
// One warp waits, with the kernels' bounded wait, on a barrier that nothing arrives at: the wait runs out
// after its cycle limit (about half a second), records the expiry and the kernel returns by itself.
__global__ void wait_expiry_selftest_kernel(unsigned int* status) {
  __shared__ uint64_t bar;
  __shared__ attn::AbortCell abort_cell;
  if (threadIdx.x == 0) {
    attn::abort_cell_init(&abort_cell, status);
    sm100::mbar_init(sm100::smem_u32(&bar), 1);
    sm100::fence_mbar_init();
  }
  __syncthreads();
  (void)attn::wait_bar_warp(sm100::smem_u32(&bar), 0, &abort_cell.flag,
                            attn::wait_info(attn::kRoleSimple, attn::kBarSync, ATTN_SELFTEST_STEP));
}

// The other way out of a wait: a warp with a copy under way waits with wait_quiet on a barrier that nothing arrives at, drains
// its copy, and one thread reports.  The reported step is ATTN_SELFTEST_STEP only if the copy had landed when its drain
// ended, and a drain of the barrier that nothing arrives at gave up.
__device__ __align__(16) uint32_t g_selftest_words[4] = {0x11, 0x22, 0x33, 0x44};
__global__ void quiet_expiry_selftest_kernel(unsigned int* status) {
  __shared__ uint64_t bar, copy_bar;
  __shared__ __align__(16) uint32_t words[4];
  __shared__ attn::AbortCell abort_cell;
  if (threadIdx.x == 0) {
    attn::abort_cell_init(&abort_cell, status);
    sm100::mbar_init(sm100::smem_u32(&bar), 1);
    sm100::mbar_init(sm100::smem_u32(&copy_bar), 1);
    sm100::fence_mbar_init();
    sm100::mbar_arrive_expect_tx(sm100::smem_u32(&copy_bar), sizeof words);
    sm100::bulk_load(sm100::smem_u32(words), g_selftest_words, sizeof words, sm100::smem_u32(&copy_bar));
  }
  __syncthreads();
  const bool arrived = attn::wait_quiet_warp(sm100::smem_u32(&bar), 0, &abort_cell.flag,
                                             attn::wait_info(attn::kRoleSimple, attn::kBarSync, ATTN_SELFTEST_STEP));
  if (!arrived && threadIdx.x == 0) {
    bool good = attn::drain_bar(sm100::smem_u32(&copy_bar), 0);
    for (int i = 0; i < 4; ++i) good = good && words[i] == g_selftest_words[i];
    good = good && !attn::drain_bar(sm100::smem_u32(&bar), 0);
    if (!good) abort_cell.info = attn::wait_info(attn::kRoleSimple, attn::kBarSync, 0);
  }
  __syncthreads();
  if (threadIdx.x == 0) attn::report_abort(&abort_cell);
}

// The way out of wait_on, as a warp that issues products takes it: a phase that nothing completes runs out, the wait after it ends at once,
// no lane may issue or pass anything on, and the warp finds out when it looks.  A second warp whose phase has completed issues a product,
// by one lane, and drains it: its accumulator, 128 x 128 sums of 64 ones, is complete then.  The reported step is ATTN_SELFTEST_STEP only
// if all of that was so.
__global__ void issue_expiry_selftest_kernel(unsigned int* status) {
  __shared__ __align__(1024) uint32_t ones[2][128 * 32];           // two tiles of [128][64] bf16
  __shared__ uint64_t bar, done_bar, drained;
  __shared__ attn::AbortCell abort_cell;
  __shared__ int issued[2], seen, wrong;
  __shared__ uint32_t tmem_slot;
  const int warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    attn::abort_cell_init(&abort_cell, status);
    sm100::mbar_init(sm100::smem_u32(&bar), 1);
    sm100::mbar_init(sm100::smem_u32(&done_bar), 1);
    sm100::fence_mbar_init();
    sm100::mbar_arrive(sm100::smem_u32(&done_bar));
    issued[0] = issued[1] = seen = wrong = 0;
  }
  for (int i = threadIdx.x; i < 2 * 128 * 32; i += blockDim.x) (&ones[0][0])[i] = 0x3F803F80u;
  sm100::fence_proxy_async_smem();
  if (warp == 1) {
    sm100::tmem_alloc(sm100::smem_u32(&tmem_slot), 128);
    sm100::tmem_relinquish();
  }
  sm100::tc_fence_before();
  __syncthreads();
  sm100::tc_fence_after();
  const uint32_t info = attn::wait_info(attn::kRoleSimple, attn::kBarSync, ATTN_SELFTEST_STEP);
  bool dead = false;
  attn::wait_on(sm100::smem_u32(warp == 0 ? &bar : &done_bar), 0, &abort_cell.flag, info, dead);
  const long long t0 = clock64();
  if (warp == 0) attn::wait_on(sm100::smem_u32(&bar), 0, &abort_cell.flag, info, dead);
  const bool quick = clock64() - t0 < attn::kWaitLimitCycles / 16;
  if (attn::may_issue(dead)) {
    atomicAdd(&issued[warp], 1);
    if (warp == 1) {
      attn::issue_qk<64, 128>(tmem_slot, sm100::smem_u32(ones[0]), sm100::smem_u32(ones[1]));
      if (!attn::drain_products(sm100::smem_u32(&drained))) atomicAdd(&wrong, 1);
    }
  }
  __syncwarp();
  if (warp == 1) {
    sm100::tc_fence_after();
    for (int c = 0; c < 4; ++c) {
      uint32_t r[32];
      sm100::tmem_ld32(tmem_slot + (32u << 16) + c * 32, r);       // (rows 32 to 63: warp 1's)
      for (int k = 0; k < 32; ++k)
        if (r[k] != __float_as_uint(64.0f)) atomicAdd(&wrong, 1);
    }
    sm100::tc_fence_before();
    __syncwarp();
    sm100::tmem_dealloc(tmem_slot, 128);
  }
  if (attn::any_dead(dead) && dead && quick) atomicAdd(&seen, 1);
  __syncthreads();
  if (threadIdx.x == 0) {
    if (issued[0] != 0 || issued[1] != 1 || seen != 32 || wrong != 0) abort_cell.info = attn::wait_info(attn::kRoleSimple, attn::kBarSync, 0);
    attn::report_abort(&abort_cell);
  }
}
}  // namespace

namespace {
template <class Kernel>
int launch_selftest(Kernel kern, uint32_t* status_dev, void* cuda_stream, int threads = 32) {
  if (status_dev && ((uintptr_t)status_dev & 15u)) return ATTN_ERR_MISALIGNED;
  DeviceState* st = nullptr;
  int rc = device_state(&st);
  if (rc != ATTN_OK) return rc;
  kern<<<1, threads, 0, static_cast<cudaStream_t>(cuda_stream)>>>(status_dev);
  ATTN_CUDA_TRY(cudaGetLastError());
  return ATTN_OK;
}
}  // namespace

extern "C" int attn_selftest_wait_expiry_to(uint32_t* status_dev, void* cuda_stream) {
  return launch_selftest(wait_expiry_selftest_kernel, status_dev, cuda_stream);
}

extern "C" int attn_selftest_quiet_expiry_to(uint32_t* status_dev, void* cuda_stream) {
  return launch_selftest(quiet_expiry_selftest_kernel, status_dev, cuda_stream);
}

extern "C" int attn_selftest_issue_expiry_to(uint32_t* status_dev, void* cuda_stream) {
  return launch_selftest(issue_expiry_selftest_kernel, status_dev, cuda_stream, 64);
}

extern "C" int attn_selftest_wait_expiry(void* cuda_stream) { return attn_selftest_wait_expiry_to(nullptr, cuda_stream); }

extern "C" int attn_last_device_status(void* cuda_stream, uint32_t* detail) {
  ATTN_CUDA_TRY(cudaStreamSynchronize(static_cast<cudaStream_t>(cuda_stream)));
  unsigned int h[4] = {0, 0, 0, 0};
  ATTN_CUDA_TRY(cudaMemcpyFromSymbol(h, attn::g_attn_dev_status, sizeof h));
  if (detail)
    for (int i = 0; i < 4; ++i) detail[i] = h[i];
  if (h[0] == 0) return ATTN_OK;
  unsigned int z[4] = {0, 0, 0, 0};
  ATTN_CUDA_TRY(cudaMemcpyToSymbol(attn::g_attn_dev_status, z, sizeof z));
  {
    // an aborted launch may have left arrival counters non-zero
    int dev = 0;
    ATTN_CUDA_TRY(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lk(g_mu);
    if (dev >= 0 && dev < kMaxDevices && g_dev[dev].ws && g_dev[dev].ws_bytes >= (size_t)attn::kCounterBytes)
      ATTN_CUDA_TRY(cudaMemset(g_dev[dev].ws, 0, attn::kCounterBytes));
  }
  return ATTN_ERR_DEVICE_TIMEOUT;
}

extern "C" int attn_last_launch_count(void) { return t_launch_count; }
extern "C" int attn_last_cluster_size(void) { return t_cluster_size; }
extern "C" int attn_last_kernel(void) { return t_kernel; }
extern "C" int attn_last_grid(void) { return t_grid; }
extern "C" const char* attn_last_kernel_name(void) {
  thread_local char text[96];
  const Instantiation& x = t_instantiation;
  int n = std::snprintf(text, sizeof text, "%s", x.name);
  for (int i = 0; i < x.args; ++i) n += std::snprintf(text + n, sizeof text - n, "%c%d%s", i ? ',' : '<', x.arg[i], i + 1 == x.args ? ">" : "");
  return text;
}

extern "C" const char* attn_last_cuda_error(void) { return t_cuda_error; }

extern "C" const char* attn_status_string(int status) {
  switch (status) {
    case ATTN_OK: return "ok";
    case ATTN_ERR_INVALID_ARG: return "invalid argument";
    case ATTN_ERR_UNSUPPORTED_SHAPE: return "unsupported shape (need d in {64,128})";
    case ATTN_ERR_MISALIGNED: return "device pointer not 16-byte aligned";
    case ATTN_ERR_ALIASING: return "output overlaps an input";
    case ATTN_ERR_INFEASIBLE_PLAN: return "no feasible tile plan";
    case ATTN_ERR_WRONG_ARCH: return "device is not compute capability 10.x";
    case ATTN_ERR_NEED_WORKSPACE: return "CTAs share Q tiles: register a workspace with attn_set_workspace (or pass one to attn_forward_ws)";
    case ATTN_ERR_CUDA: return "CUDA error (see attn_last_cuda_error)";
    case ATTN_ERR_DEVICE_TIMEOUT: return "a bounded device-side wait expired";
    case ATTN_ERR_BAD_TILES: return "tile override not available";
    case ATTN_ERR_SCRATCH_LIMIT: return "problem needs more scratch than the library's built-in array holds";
    default: return "unknown status";
  }
}

// ===========================================================================
// Unfused path: matrix product, row softmax, three-kernel attention
// ===========================================================================
namespace {

// 3-D map over a contiguous [batch][rows][cols] bf16 tensor with a (64 columns, box_rows rows, 1) box.
int make_tmap_mat(CUtensorMap* m, const void* base, int batch, int rows, int cols, int box_rows) {
  return make_tmap(m, base, batch, rows, cols, box_rows);
}

// Products that gemm_small_kernel takes over from the plan's kernels: at most one 128 x 128 tile per SM, where the plan's tile
// is larger.  There it is faster at every size measured (1.2 to 1.6 times where the plan has lone CTAs, 1.0 to 1.3 times where
// it has pairs; K = 64 to 8192).  A plan of 128 x 128 tiles keeps its kernel: there neither is faster at every size (us, plan /
// this, operands in the cache: 16384 x 128 x 2048 13.7 / 14.6, 128 x 128 x 8192 34.3 / 36.6, 16384 x 128 x 16384 98 / 88).  K is never shared out between CTAs: an element's
// sum would depend on how many tiles stand beside it.
bool gemm_small(int batch, int M, int N, const gemm_tiles& t, int sms) {
  const long long tiles = (long long)batch * ((M + 127) / 128) * ((N + 127) / 128);
  return tiles <= sms && (t.tile_m > 128 || t.tile_n > 128);
}

int gemm_launch(const void* a, const void* b, void* c, int batch, int M, int N, int K, int b_layout, cudaStream_t stream,
                const gemm_tiles* ovr = nullptr) {
  if (!a || !b || !c || batch <= 0 || M <= 0 || N <= 0 || K <= 0) return ATTN_ERR_INVALID_ARG;
  if (b_layout != 0 && b_layout != 1) return ATTN_ERR_INVALID_ARG;
  if ((K & 7) || (N & 7)) return ATTN_ERR_UNSUPPORTED_SHAPE;
  if (((uintptr_t)a | (uintptr_t)b | (uintptr_t)c) & 15u) return ATTN_ERR_MISALIGNED;
  const size_t a_bytes = (size_t)batch * M * K * 2, b_bytes = (size_t)batch * N * K * 2, c_bytes = (size_t)batch * M * N * 2;
  if (overlaps(c, c_bytes, a, a_bytes) || overlaps(c, c_bytes, b, b_bytes)) return ATTN_ERR_ALIASING;
  DeviceState* st = nullptr;
  int rc = device_state(&st);
  if (rc != ATTN_OK) return rc;
  gemm_tiles t;
  if (ovr) {
    // tile sweep: the derivation re-run with pairs switched off (cta_pair 1) or with the other tile width
    attn_hw_desc d2 = st->desc;
    if (ovr->cta_pair == 1) d2.max_clusters[1] = 0;
    if ((rc = gemm_plan(&d2, batch, M, N, K, &t)) != ATTN_OK) return rc;
    if (ovr->cta_pair == 2 && t.cta_pair != 2) return ATTN_ERR_BAD_TILES;
    if (ovr->tile_n > 0 && ovr->tile_n != t.tile_n) {
      if (t.cta_pair != 2 || (ovr->tile_n != 128 && ovr->tile_n != 256)) return ATTN_ERR_BAD_TILES;
      t.tile_n = ovr->tile_n;
      const int stage = gemm::pair_stage_bytes(t.tile_n);
      t.stages = std::min(gemm::kMaxStages, (st->desc.local_mem_bytes - gemm::kPairOutBytes - gemm::kMiscBytes) / stage);
      t.tiles = batch * ((M + 255) / 256) * ((N + t.tile_n - 1) / t.tile_n);
      t.ctas = 2 * std::min(t.tiles, std::min(st->desc.max_clusters[1], st->desc.num_units / 2));
      t.acc_buffers = 512 / t.tile_n;
      t.tail_split = 0;
    }
    if (ovr->tail_split < 0) t.tail_split = 0;                 // (sweep: whole tiles in the last wave too)
  } else if ((rc = gemm_plan(&st->desc, batch, M, N, K, &t)) != ATTN_OK) {
    return rc;
  }
  // the kernels are compiled for exactly the tile shapes the derivation gives on this architecture
  if (!t.feasible || (t.n_sub != 1 && t.n_sub != 2) || t.tile_m != t.n_sub * attn::kSub || (t.tile_n != 128 && t.tile_n != 256) ||
      t.tile_k != gemm::kTileK || t.stages > gemm::kMaxStages || t.stages < 2)
    return ATTN_ERR_INFEASIBLE_PLAN;
  if (!ovr && gemm_small(batch, M, N, t, st->desc.num_units)) {
    CUtensorMap ta, tb;
    if ((rc = make_tmap_mat(&ta, a, batch, M, K, 128)) != ATTN_OK) return rc;
    if (b_layout == 0) rc = make_tmap_mat(&tb, b, batch, K, N, gemm::kTileK);
    else rc = make_tmap_mat(&tb, b, batch, N, K, 128);
    if (rc != ATTN_OK) return rc;
    gemm::GemmParams p = {};
    p.M = M; p.N = N; p.K = K; p.batch = batch;
    p.m_tiles = (M + 127) / 128;
    p.n_tiles = (N + 127) / 128;
    p.k_steps = (K + gemm::kTileK - 1) / gemm::kTileK;
    p.stages = std::min(gemm::kMaxStages, (st->desc.local_mem_bytes - gemm::kMiscBytes) / gemm::kSmallStageBytes);
    const int tiles = batch * p.m_tiles * p.n_tiles, smem = gemm::small_smem_total(p.stages);
    auto launch_small = [&](auto kernel) -> int {
      ATTN_ALLOW_SMEM(kernel, smem);
      ATTN_CUDA_TRY(launch_kernel(kernel, tiles, gemm::kThreads, smem, 0, stream, ta, tb, static_cast<__nv_bfloat16*>(c), p));
      return ATTN_OK;
    };
    rc = b_layout == 0 ? launch_small(gemm::gemm_small_kernel<true>) : launch_small(gemm::gemm_small_kernel<false>);
    if (rc != ATTN_OK) return rc;
    ATTN_CUDA_TRY(cudaGetLastError());
    ++t_launch_count;
    launched(ATTN_KERNEL_GEMM_SMALL, tiles, {"gemm_small_kernel", 1, {b_layout == 0 ? 1 : 0}});
    return ATTN_OK;
  }
  CUtensorMap ta, tb, tc;
  const bool pair = t.cta_pair == 2;
  // a CTA of a pair stages its own 128 rows of A and tile_n / 2 columns (rows, for [N][K]) of B
  if ((rc = make_tmap_mat(&ta, a, batch, M, K, attn::kSub)) != ATTN_OK) return rc;
  if (b_layout == 0) rc = make_tmap_mat(&tb, b, batch, K, N, gemm::kTileK);    // [K][N]: box 64 columns x 64 k-rows
  else rc = make_tmap_mat(&tb, b, batch, N, K, pair ? t.tile_n / 2 : t.tile_n);   // [N][K]: box 64 k-columns x rows of B
  if (rc != ATTN_OK) return rc;
  // (a pair's epilogue warps each store their own 32 rows)
  if ((rc = make_tmap_mat(&tc, c, batch, M, N, pair ? 32 : attn::kSub)) != ATTN_OK) return rc;
  gemm::GemmParams p;
  p.M = M; p.N = N; p.K = K; p.batch = batch;
  p.n_sub = t.n_sub;
  p.m_tiles = (M + t.tile_m - 1) / t.tile_m;
  p.n_tiles = (N + t.tile_n - 1) / t.tile_n;
  p.k_steps = (K + gemm::kTileK - 1) / gemm::kTileK;
  p.stages = t.stages;
  p.group_m = 1;
  p.tail_tiles = 0;
  p.stream_c = (long long)batch * M * N * 2 > (long long)st->desc.cache_bytes ? 1 : 0;
  if (pair) {
    // Bands of about sqrt(pairs) tile rows: the tiles in flight then share the fewest operand panels.  Only when the
    // operands of a tile outweigh its output eightfold (K >= 1024 for 256 x 256 tiles): below that the output
    // dominates the traffic, and tile rows walked whole write whole rows of C (16384 x 16384 x 64: 141 against 156 us).
    const int pairs = t.ctas / 2;
    int gm = 1;
    if ((long long)(t.tile_m + t.tile_n) * K >= 8LL * t.tile_m * t.tile_n)
      while ((gm + 1) * (gm + 1) <= pairs) ++gm;
    p.group_m = gm;
    p.tail_tiles = t.tail_split;
    const int smem = gemm::pair_smem_total(t.stages, t.tile_n);
    auto launch_pair = [&](auto kernel) -> int {
      ATTN_ALLOW_SMEM(kernel, smem);
      ATTN_CUDA_TRY(launch_kernel(kernel, t.ctas, gemm::kPairThreads, smem, 2, stream, ta, tb, tc, p));
      return ATTN_OK;
    };
    if (t.tile_n == 256) rc = (b_layout == 0) ? launch_pair(gemm::gemm_pair_kernel<true, 256>) : launch_pair(gemm::gemm_pair_kernel<false, 256>);
    else rc = (b_layout == 0) ? launch_pair(gemm::gemm_pair_kernel<true, 128>) : launch_pair(gemm::gemm_pair_kernel<false, 128>);
  } else {
    const int smem = gemm::smem_total(t.stages, t.tile_n);
    auto launch = [&](auto kernel) -> int {
      ATTN_ALLOW_SMEM(kernel, smem);
      ATTN_CUDA_TRY(launch_kernel(kernel, t.ctas, gemm::kThreads, smem, 0, stream, ta, tb, tc, p));
      return ATTN_OK;
    };
    if (t.tile_n == 256) rc = (b_layout == 0) ? launch(gemm::gemm_kernel<true, 256>) : launch(gemm::gemm_kernel<false, 256>);
    else rc = (b_layout == 0) ? launch(gemm::gemm_kernel<true, 128>) : launch(gemm::gemm_kernel<false, 128>);
  }
  if (rc != ATTN_OK) return rc;
  ATTN_CUDA_TRY(cudaGetLastError());
  ++t_launch_count;
  launched(pair ? ATTN_KERNEL_GEMM_PAIR : ATTN_KERNEL_GEMM, t.ctas, {pair ? "gemm_pair_kernel" : "gemm_kernel", 2, {b_layout == 0 ? 1 : 0, t.tile_n}});
  return ATTN_OK;
}

int softmax_launch(const void* s, void* pout, long long rows, int cols, float scale, cudaStream_t stream) {
  // the kernels take the row maximum on the raw scores and scale it afterwards: the scale must keep the order
  if (!s || !pout || rows <= 0 || cols <= 0 || !(scale > 0.0f) || !std::isfinite(scale)) return ATTN_ERR_INVALID_ARG;
  if ((cols & 7) || cols > 32768 || rows > 0x7FFFFFFFLL) return ATTN_ERR_UNSUPPORTED_SHAPE;
  if (((uintptr_t)s | (uintptr_t)pout) & 15u) return ATTN_ERR_MISALIGNED;
  const float scale_log2 = scale * 1.4426950408889634f;
  const int nvec = cols / 8;                        // 16-byte vectors per row
  const __nv_bfloat16* sp = static_cast<const __nv_bfloat16*>(s);
  __nv_bfloat16* pp = static_cast<__nv_bfloat16*>(pout);
  DeviceState* st = nullptr;
  int rc = device_state(&st);
  if (rc != ATTN_OK) return rc;
  const int sms = st->desc.num_units;
  long long ctas = rows;
  // Up to 128 vectors a row: a warp per row (half a warp below 17 vectors), at most 16 CTAs of four warps per SM
  // (65536 x 1024: 43.2 us, 8 CTAs 47.9; one CTA per row is slower at every width up to here).
  auto launch_warp = [&](auto kern, int rows_per_warp) {
    ctas = std::min((rows + 4 * rows_per_warp - 1) / (4 * rows_per_warp), 16LL * sms);
    return launch_kernel(kern, ctas, 128, 0, 0, stream, sp, pp, rows, cols, scale_log2);
  };
  // Longer rows: a CTA per row, as few warps as hold it at VPT vectors a thread (5000 columns on 160 threads: 16.9 us for
  // 5000 rows; a kernel with 256 threads for every row of 4104 to 8192 columns took 24.6).  Their CTAs let the next grid in when they
  // end: let in earlier, its CTAs are in the way of those of this one (us in graphs, early / at the end: 10000 x 1032 11.6 / 7.8,
  // 32768 x 1032 35.6 / 24.8, 256 x 32768 10.7 / 7.8, 1000 x 4096 3.7 / 3.4; the same beyond 2000 x 4096).
  auto launch_row = [&](auto kern, int threads) { return launch_kernel(kern, rows, threads, 0, 0, stream, sp, pp, cols, scale_log2); };
#define SOFTMAX_ROW_CASE(VPT_, THREADS_) else if (nvec <= VPT_ * THREADS_) e = launch_row(gemm::softmax_rows_kernel<VPT_, THREADS_>, THREADS_)
  cudaError_t e = cudaSuccess;
  if (nvec <= 16) e = launch_warp(gemm::softmax_rows_warp_kernel<1, 16>, 2);
  else if (nvec <= 32) e = launch_warp(gemm::softmax_rows_warp_kernel<1, 32>, 1);
  else if (nvec <= 64) e = launch_warp(gemm::softmax_rows_warp_kernel<2, 32>, 1);
  else if (nvec <= 96) e = launch_warp(gemm::softmax_rows_warp_kernel<3, 32>, 1);
  else if (nvec <= 128) e = launch_warp(gemm::softmax_rows_warp_kernel<4, 32>, 1);
  SOFTMAX_ROW_CASE(2, 96);
  SOFTMAX_ROW_CASE(2, 128);
  SOFTMAX_ROW_CASE(4, 96);
  SOFTMAX_ROW_CASE(4, 128);
  SOFTMAX_ROW_CASE(4, 160);
  SOFTMAX_ROW_CASE(4, 192);
  SOFTMAX_ROW_CASE(4, 224);
  SOFTMAX_ROW_CASE(4, 256);
  SOFTMAX_ROW_CASE(8, 160);
  SOFTMAX_ROW_CASE(8, 192);
  SOFTMAX_ROW_CASE(8, 224);
  SOFTMAX_ROW_CASE(8, 256);
  else {
    // wider than the registers of one block hold: the row is staged in shared memory (2 bytes per column)
    auto kern = gemm::softmax_rows_staged_kernel<256>;
    ATTN_ALLOW_SMEM(kern, 65536);
    e = launch_kernel(kern, rows, 256, cols * 2, 0, stream, sp, pp, cols, scale_log2);
  }
#undef SOFTMAX_ROW_CASE
  ATTN_CUDA_TRY(e);
  ++t_launch_count;
  launched(ATTN_KERNEL_SOFTMAX, ctas, {"softmax_rows", 0, {}});
  return ATTN_OK;
}

}  // namespace

extern "C" int gemm_forward(const void* a, const void* b, void* c, int batch, int M, int N, int K, int b_layout,
                            void* cuda_stream) {
  t_launch_count = 0;
  return gemm_launch(a, b, c, batch, M, N, K, b_layout, static_cast<cudaStream_t>(cuda_stream));
}

extern "C" int gemm_forward_call(const gemm_call* g) {
  if (!g) return ATTN_ERR_INVALID_ARG;
  return gemm_forward(g->a, g->b, g->c, g->batch, g->M, g->N, g->K, g->b_layout, g->cuda_stream);
}

extern "C" int softmax_rows_forward_call(const softmax_call* c) {
  if (!c) return ATTN_ERR_INVALID_ARG;
  return softmax_rows_forward(c->s, c->p, c->rows, c->cols, (float)c->scale, c->cuda_stream);
}

extern "C" int gemm_forward_tiles(const void* a, const void* b, void* c, int batch, int M, int N, int K, int b_layout,
                                  const gemm_tiles* override_tiles, void* cuda_stream) {
  t_launch_count = 0;
  return gemm_launch(a, b, c, batch, M, N, K, b_layout, static_cast<cudaStream_t>(cuda_stream), override_tiles);
}

extern "C" int softmax_rows_forward(const void* s, void* p, long long rows, int cols, float scale, void* cuda_stream) {
  t_launch_count = 0;
  return softmax_launch(s, p, rows, cols, scale, static_cast<cudaStream_t>(cuda_stream));
}

extern "C" int attn_forward_unfused(const void* q, const void* k, const void* v, void* o, void* scores, size_t scores_bytes,
                                    int B, int H, int L, int d, void* cuda_stream) {
  t_launch_count = 0;
  if (!q || !k || !v || !o || !scores || B <= 0 || H <= 0 || L <= 0 || d <= 0) return ATTN_ERR_INVALID_ARG;
  if ((L & 7) || (d & 7) || L > 32768) return ATTN_ERR_UNSUPPORTED_SHAPE;
  const size_t need = (size_t)B * H * L * L * 2;
  if (scores_bytes < need) return ATTN_ERR_INVALID_ARG;
  const size_t bytes = (size_t)B * H * L * d * 2;
  if (overlaps(o, bytes, q, bytes) || overlaps(o, bytes, k, bytes) || overlaps(o, bytes, v, bytes)) return ATTN_ERR_ALIASING;
  if (overlaps(scores, need, q, bytes) || overlaps(scores, need, k, bytes) || overlaps(scores, need, v, bytes) ||
      overlaps(scores, need, o, bytes))
    return ATTN_ERR_ALIASING;
  cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
  int rc;
  if ((rc = gemm_launch(q, k, scores, B * H, L, L, d, 1, stream)) != ATTN_OK) return rc;           // S = Q K^T
  if ((rc = softmax_launch(scores, scores, (long long)B * H * L, L, 1.0f / std::sqrt((float)d), stream)) != ATTN_OK)
    return rc;                                                                                      // P = softmax(S / sqrt(d))
  return gemm_launch(scores, v, o, B * H, L, d, L, 0, stream);                                      // O = P V
}
