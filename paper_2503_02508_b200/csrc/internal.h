// Internal declarations shared by the translation units of libqdit (not part of the C ABI).
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <unordered_map>
#include <unordered_set>
#include <vector>

#include "qdit.h"

// Device status word values (written by kernels, read by qdit_sync).
enum : int { QDIT_DEV_OK = 0, QDIT_DEV_TIMEOUT = 1 };

struct TmapKey {
  const void* ptr;
  uint64_t rows, cols, ld;
  uint32_t box_rows, box_cols, swizzle, esize;
  bool operator==(const TmapKey& o) const {
    return ptr == o.ptr && rows == o.rows && cols == o.cols && ld == o.ld && box_rows == o.box_rows &&
           box_cols == o.box_cols && swizzle == o.swizzle && esize == o.esize;
  }
};
struct TmapKeyHash {
  size_t operator()(const TmapKey& k) const {
    uint64_t h = reinterpret_cast<uint64_t>(k.ptr);
    auto mix = [&](uint64_t v) { h ^= v + 0x9E3779B97F4A7C15ull + (h << 6) + (h >> 2); };
    mix(k.rows); mix(k.cols); mix(k.ld); mix(k.box_rows); mix(k.box_cols); mix(k.swizzle); mix(k.esize);
    return static_cast<size_t>(h);
  }
};

struct qdit_ctx {
  int device = 0;
  cudaStream_t stream = nullptr;
  int* d_status = nullptr;  // device status word
  int* h_status = nullptr;  // pinned host mirror
  int num_sms = 0;
  int64_t launches = 0;
  // Kernel-selection options (qdit_set_option).  Set once at creation from the QDIT_* environment variables of the
  // same names, afterwards only through the call; no kernel launch reads the environment.
  int opt[QDIT_OPT_COUNT] = {};
  bool overlap_launches = true;  // = opt[QDIT_OPT_PDL]: programmatic dependent launch for the kernels that support it
  std::unordered_set<const void*> attr_done;  // kernels whose dynamic shared-memory limit has been raised for this context
  std::string last_error;
  int sk_clusters[8] = {};    // split-reduction GEMM: clusters of that many CTAs resident at once (0 = not asked yet)
  void* encode_fn = nullptr;  // cuTensorMapEncodeTiled
  std::unordered_map<TmapKey, CUtensorMap, TmapKeyHash> tmaps;
  // per-kernel event timing (qdit_profile_*)
  bool profiling = false;
  struct ProfRec { int kind; double work; cudaEvent_t start, stop; };
  std::vector<ProfRec> prof;
  std::vector<cudaEvent_t> event_pool;
};

// Records a formatted message on the context and returns `code`.
int32_t qdit_fail(qdit_ctx* ctx, int32_t code, const char* fmt, ...);

// Brackets one kernel launch with events while profiling is enabled.
struct ProfScope {
  qdit_ctx* ctx;
  bool on;
  cudaEvent_t stop;
  ProfScope(qdit_ctx* c, int kind, double work);
  ~ProfScope();
};

// Launches `kernel` on the context's stream.  With ctx->overlap_launches the launch carries the
// programmatic-stream-serialization attribute: the kernel may start its preamble before the previous kernel
// of the stream has finished, and MUST call grid_dependency_wait() before its first access to global memory that an earlier
// launch of the stream may write (weights that are constant since the model was created may be fetched before).
// What a launch of this library may write just in front is not read through the read-only path (`__ldg`, or a `const __restrict__`
// parameter), which is defined for data that do not change while the kernel lives.  The rows of the LayerNorm and of the per-token
// quantizer still are, behind grid_dependency_wait(): without it their loops' loads stay behind the stores of the pass before (640 x 8192
// f32 per token 9.9 / 12.5 us); so is the scale of the LayerNorm of any width (without it 80 registers instead of 64, 8192 x 392 f32 5.8 / 6.9).
template <typename... KArgs, typename... Args>
cudaError_t qdit_launch_overlapped(qdit_ctx* ctx, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                                   Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = ctx->stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = ctx->overlap_launches ? 1 : 0;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// The same with thread-block clusters of `cluster` CTAs (the grid is a multiple of it).
template <typename... KArgs, typename... Args>
cudaError_t qdit_launch_cluster(qdit_ctx* ctx, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, unsigned cluster,
                                Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = ctx->stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = ctx->overlap_launches ? 1 : 0;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = cluster;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// Raises a kernel's dynamic shared-memory limit once per context (the attribute is per device and function; a context
// belongs to one device and is used by one thread at a time, so no process-wide state is involved).
template <typename K>
int32_t qdit_allow_smem(qdit_ctx* ctx, K kernel, int bytes) {
  const void* key = reinterpret_cast<const void*>(kernel);
  if (ctx->attr_done.count(key)) return QDIT_OK;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e != cudaSuccess) return qdit_fail(ctx, QDIT_ERR_CUDA, "cudaFuncSetAttribute: %s", cudaGetErrorString(e));
  ctx->attr_done.insert(key);
  return QDIT_OK;
}

// Checks the last launch; counts it.
int32_t qdit_after_launch(qdit_ctx* ctx, const char* what);

#define QDIT_CUDA_CHECK(ctx, expr)                                                                             \
  do {                                                                                                         \
    cudaError_t e__ = (expr);                                                                                  \
    if (e__ != cudaSuccess) return qdit_fail((ctx), QDIT_ERR_CUDA, "%s: %s", #expr, cudaGetErrorString(e__)); \
  } while (0)
#define QDIT_TRY(expr)                 \
  do {                                 \
    int32_t st__ = (expr);             \
    if (st__ != QDIT_OK) return st__;  \
  } while (0)

// 2-D tensor map over a row-major matrix [rows, cols] of `esize`-byte elements with row pitch `ld`
// elements; box = box_rows x box_cols elements; swizzle: 0 none, 1 = 128-byte, 2 = 64-byte, 3 = 32-byte.
// Cached per context.
int32_t qdit_get_tmap(qdit_ctx* ctx, const void* ptr, uint64_t rows, uint64_t cols, uint64_t ld, uint32_t box_rows,
                      uint32_t box_cols, uint32_t swizzle, uint32_t esize, CUtensorMap* out);

// Quantizer parameters as the kernels take them.
struct QuantArgs {
  float scale;             // s (by value)
  const float* scale_dev;  // if non-null, overrides `scale`
  float zp, qmin, qmax;    // as floats (exact small integers)
};
inline QuantArgs make_quant_args(const qdit_qparams& qp, const float* scale_dev) {
  QuantArgs a;
  a.scale = qp.scale;
  a.scale_dev = scale_dev;
  a.zp = static_cast<float>(qp.zero_point);
  a.qmin = static_cast<float>(qp.qmin);
  a.qmax = static_cast<float>(qp.qmax);
  return a;
}
int32_t qdit_check_qparams(qdit_ctx* ctx, const qdit_qparams* qp, bool scale_from_device);

static inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// ---- internal launchers used by the model/sampler orchestration (all enqueue on ctx->stream) ----
// Dynamic symmetric quantizer of a whole tensor: codes, the scale in *scale (required), max|x| folded into *running (optional).
// Works in q and *scale alone.
int32_t launch_quant_dynamic(qdit_ctx* ctx, const void* x, int x_dtype, int64_t M, int64_t K, int64_t ldx, float* scale, float* running,
                             void* q, int64_t ldq);
int32_t launch_absmax_to_scale(qdit_ctx* ctx, const float* absmax_dev, float* scale_dev, int n);
// Quantizes an f32 tensor [M,K] (contiguous) with the scale held in device memory.
int32_t qdit_quantize_act_dev(qdit_ctx* ctx, const float* x, int64_t M, int64_t K, qdit_qparams qp,
                              const float* scale_dev, uint8_t* q);
// qdit_w8a8_linear (or qdit_w4a8_linear: packed4) for the model's own layers, whose weights (`early`), weight scales, biases, gates and
// quantizer scales (`early_params`) were written at least two launches ago.  In this and the next two calls `absmax`, if given, takes the largest magnitude of an f32 output.
int32_t qdit_linear_impl(qdit_ctx* ctx, const void* A, const void* W, int64_t M, int64_t N, int64_t K, qdit_qparams a_qp,
                         const float* a_scale_dev, uint32_t flags, const qdit_epilogue* epi, void* out, int64_t ldo, bool packed4,
                         void* w8_scratch, bool early, bool early_params, float* absmax = nullptr);
// qdit_adaln_modulate; `early`: modulation and scale were written at least two launches ago (both kernels of a pair of launches may be
// resident at once, but every kernel lets its successor start only after its own wait, so the launch before the previous one is complete)
int32_t qdit_adaln_impl(qdit_ctx* ctx, const void* x, int64_t M, int64_t D, int64_t T, float eps, const float* shift, const float* scale,
                        int64_t ld_mod, void* out, int out_dtype, const qdit_qparams* out_qp, const float* out_scale_dev, bool early, float* absmax = nullptr);
int32_t qdit_attention_impl(qdit_ctx* ctx, const void* q, const void* k, const void* v, int64_t ld, int B, int H, int T, int dh, float softmax_scale,
                            void* out, int out_dtype, const qdit_qparams* out_qp, const float* out_scale_dev, float* absmax);
// The quantizer behind one of these calls whose f32 output's largest magnitude went to *absmax (which was zero before): codes, the scale
// in *scale, the magnitude folded into *running; x contiguous, K % 16 == 0.
int32_t launch_quant_absmax(qdit_ctx* ctx, const float* x, int64_t M, int64_t K, const float* absmax, float* scale, float* running, void* q);
