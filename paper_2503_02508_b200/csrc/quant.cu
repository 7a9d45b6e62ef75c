// HBM-bound quantizer kernels: activation quantizer (Eq. 1), abs-max reduction for dynamic ranges,
// channel-wise weight quantizer, and LayerNorm + adaLN modulation with the fused activation quantizer.
#include "common.cuh"
#include "internal.h"

namespace {

using namespace qd;

// Quantizers of few CTAs start before the kernel in front of them has ended.  More of them would be packed onto the SMs that this kernel
// leaves free, eight to an SM, and those set the pace when it is over: per-token quantizer and layer, 1024 x 1152 x 4608 (128 CTAs)
// 35.6 us started early, 22.5 not; 512 rows (64) 21.8 and 14.2; 256 rows (32) 12.8 and 13.4.  The static one has a fourth of that work
// per CTA: 2048 x 3456 x 1152 (576 CTAs) 14.3 and 13.5, 512 rows (144) 8.5 and 7.9, 64 x 1152 x 4608 (72) 7.9 and 8.8.
constexpr unsigned EARLY_CTAS = 128, EARLY_TOKEN_CTAS = 48;
// A static quantizer of more CTAs than this does not let its successor start early either (64417 x 4608 x 1152, 18000 CTAs, quantizer
// and layer: 478 us with it, 458 without; 64417 x 3456 x 1152: 362 and 350; no difference from 1000 to 4600 CTAs).
constexpr unsigned RELEASE_CTAS = 4096;

// ----------------------------------------------------------------------------- activation quantizer
// One thread per 16 consecutive elements of a row (two 8-element halves); K % 8 == 0.
template <typename T>
__global__ void __launch_bounds__(256) act_quant_kernel(const T* x, int64_t M, int64_t K, int64_t ldx,
                                                        QuantArgs qa, uint8_t* __restrict__ q, int64_t ldq) {
  grid_dependency_wait();
  if (gridDim.x <= RELEASE_CTAS) grid_dependency_release();
  const int64_t chunks_per_row = (K + 15) / 16;
  const int64_t idx = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (idx >= M * chunks_per_row) return;
  const int64_t row = idx / chunks_per_row;
  const int64_t col = (idx - row * chunks_per_row) * 16;
  const float scale = device_value(qa.scale_dev, qa.scale);
  const float inv = __fdiv_rn(1.0f, scale);
  const T* src = x + row * ldx + col;
  uint8_t* dst = q + row * ldq + col;
  const bool second = col + 8 < K;
  float a[8], b[8];
  Load8<T>::load(src, a);
  if (second) Load8<T>::load(src + 8, b);
  const uint2 lo = quantize_pack8(a, inv, qa.zp, qa.qmin, qa.qmax);
  if (second) {
    const uint2 hi = quantize_pack8(b, inv, qa.zp, qa.qmin, qa.qmax);
    if ((reinterpret_cast<uintptr_t>(dst) & 15u) == 0) {
      *reinterpret_cast<uint4*>(dst) = make_uint4(lo.x, lo.y, hi.x, hi.y);
    } else {
      *reinterpret_cast<uint2*>(dst) = lo;
      *reinterpret_cast<uint2*>(dst + 8) = hi;
    }
  } else {
    *reinterpret_cast<uint2*>(dst) = lo;
  }
}

// 8 consecutive values as they lie in memory.
template <typename T>
struct Raw8;
template <>
struct Raw8<__nv_bfloat16> {
  uint4 w;
  __device__ __forceinline__ void load(const __nv_bfloat16* p) { w = *reinterpret_cast<const uint4*>(p); }
  __device__ __forceinline__ void clear() { w = make_uint4(0u, 0u, 0u, 0u); }
  __device__ __forceinline__ void widen(float (&v)[8]) const {
    unpack_bf16x2(w.x, v[0], v[1]);
    unpack_bf16x2(w.y, v[2], v[3]);
    unpack_bf16x2(w.z, v[4], v[5]);
    unpack_bf16x2(w.w, v[6], v[7]);
  }
};
template <>
struct Raw8<float> {
  float4 a, b;
  __device__ __forceinline__ void load(const float* p) {
    a = *reinterpret_cast<const float4*>(p);
    b = *reinterpret_cast<const float4*>(p + 4);
  }
  __device__ __forceinline__ void clear() { a = b = make_float4(0.0f, 0.0f, 0.0f, 0.0f); }
  __device__ __forceinline__ void widen(float (&v)[8]) const {
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
  }
};

// Per-token dynamic quantizer: one warp per row finds max|x| of its row, s[m] = max / 127 (1 for a zero row),
// and writes the symmetric codes.
//
// Bound by memory, if enough of it is in flight: with NV > 0 a lane loads its NV pieces of 8 values at once and keeps them for
// the codes (K <= 256 * NV).  NV = 0: any K, the row is read twice, the second time from L1 / L2.
template <typename T, int NV>
__global__ void __launch_bounds__(256) act_quant_token_kernel(const T* __restrict__ x, int64_t M, int64_t K, int64_t ldx,
                                                              float* __restrict__ scales, uint8_t* __restrict__ q,
                                                              int64_t ldq) {
  grid_dependency_wait();
  grid_dependency_release();
  const int lane = threadIdx.x & 31;
  const int64_t row = static_cast<int64_t>(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (row >= M) return;
  const T* src = x + row * ldx;
  Raw8<T> raw[NV > 0 ? NV : 1];
  float m = 0.0f;
  auto widest = [&](const Raw8<T>& r) {
    float v[8];
    r.widen(v);
#pragma unroll
    for (int i = 0; i < 8; ++i) m = fmaxf(m, fabsf(v[i]));
  };
  if constexpr (NV > 0) {
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const int k = lane * 8 + i * 256;
      if (k < K) raw[i].load(src + k);
      else raw[i].clear();
    }
#pragma unroll
    for (int i = 0; i < NV; ++i) widest(raw[i]);
  } else {
    for (int64_t k = lane * 8; k < K; k += 256) {
      raw[0].load(src + k);
      widest(raw[0]);
    }
  }
  m = warp_max(m);
  float s = __fdiv_rn(m, 127.0f);
  if (!(s > 0.0f)) s = 1.0f;
  const float inv = __fdiv_rn(1.0f, s);
  if (lane == 0) scales[row] = s;
  uint8_t* dst = q + row * ldq;
  float v[8];
  if constexpr (NV > 0) {
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const int k = lane * 8 + i * 256;
      raw[i].widen(v);
      if (k < K) *reinterpret_cast<uint2*>(dst + k) = quantize_pack8(v, inv, 0.0f, -127.0f, 127.0f);
    }
  } else {
    for (int64_t k = lane * 8; k < K; k += 256) {
      raw[0].load(src + k);
      raw[0].widen(v);
      *reinterpret_cast<uint2*>(dst + k) = quantize_pack8(v, inv, 0.0f, -127.0f, 127.0f);
    }
  }
}

// ----------------------------------------------------------------------------- dynamic quantizer
// Two launches, which is what the time of a small tensor consists of (64 x 1152: 8.3 us with four, 3.2 with two): partial
// maxima, one per CTA, and a quantizer whose CTAs all reduce them.  The partials lie in the output itself, which the codes
// overwrite: memory of the call alone, whatever else runs beside it (a captured launch replayed on another stream as well).  Every
// quantizer CTA has a copy of its own, in the part of the output that it is about to write, because no other part is safe from
// being overwritten first.  A tensor of more than DYN_PIECES has one copy, at the front, and a launch of one CTA between that
// reads it before the plain quantizer starts (4300 x 1152, bf16: 9.5 us).
//
// The output in pieces of 8 codes (two floats): parts of `size` pieces, the last two of equal length, so that none is shorter than
// half of it and its partials fit.
constexpr int DYN_PARTIALS = 256;        // most CTAs that form partial maxima when every part has a copy
constexpr int64_t DYN_PIECES = 600000;
__device__ __forceinline__ int64_t part_first(int64_t total, int parts, int size, int c) {
  if (c == 0) return 0;
  return c < parts - 1 ? static_cast<int64_t>(c) * size : c == parts ? total : (static_cast<int64_t>(parts - 2) * size + total) / 2;
}
// Row of a piece of such a tensor without a division: per_row_inv = ceil(2^40 / per_row) (exact for piece * per_row < 2^40), or 0 if
// all pieces lie in row 0.
inline uint64_t inverse_of(int64_t per_row) { return per_row > DYN_PIECES ? 0 : ((1ull << 40) + per_row - 1) / per_row; }
__device__ __forceinline__ uint32_t row_of(uint32_t piece, uint64_t per_row_inv) { return static_cast<uint32_t>(piece * per_row_inv >> 40); }
__device__ __forceinline__ float* partial_at(uint8_t* q, int64_t ldq, uint32_t per_row, uint64_t per_row_inv, int64_t first, int i) {
  const uint32_t piece = static_cast<uint32_t>(first) + (i >> 1), row = row_of(piece, per_row_inv);
  return reinterpret_cast<float*>(q + static_cast<int64_t>(row) * ldq + (piece - row * per_row) * 8) + (i & 1);
}

template <typename T, int THREADS>
__global__ void __launch_bounds__(THREADS) absmax_partial_kernel(const T* x, int64_t M, int64_t K, int64_t ldx,
                                                                 uint8_t* __restrict__ q, int64_t ldq, uint64_t per_row_inv, int copies, int size) {
  grid_dependency_wait();
  grid_dependency_release();
  const int64_t vec_per_row = K / 8;
  const int64_t total = M * vec_per_row;
  float m = 0.0f;
  for (int64_t idx = static_cast<int64_t>(blockIdx.x) * THREADS + threadIdx.x; idx < total;
       idx += static_cast<int64_t>(gridDim.x) * THREADS) {
    const int64_t row = total <= DYN_PIECES ? row_of(static_cast<uint32_t>(idx), per_row_inv) : idx / vec_per_row;
    const int64_t col = (idx - row * vec_per_row) * 8;
    float v[8];
    Load8<T>::load(x + row * ldx + col, v);
#pragma unroll
    for (int i = 0; i < 8; ++i) m = fmaxf(m, fabsf(v[i]));
  }
  m = warp_max(m);
  __shared__ float smax[THREADS / 32];
  if ((threadIdx.x & 31) == 0) smax[threadIdx.x >> 5] = m;
  __syncthreads();
  m = warp_max(smax[threadIdx.x & (THREADS / 32 - 1)]);
  for (int c = threadIdx.x; c < copies; c += THREADS) 
    *partial_at(q, ldq, static_cast<uint32_t>(vec_per_row), per_row_inv, part_first(total, copies, size, c), blockIdx.x) = m;
}

// The partials -> s = max / 127 (1 for an empty range); thread 0 of CTA 0 leaves it in *scale and folds the maximum into
// *running (both optional).  256 threads; on return all of them have read their partials.
__device__ __forceinline__ float scale_of_partials(uint8_t* q, int64_t ldq, uint32_t per_row, uint64_t per_row_inv, int64_t first, int n_partial,
                                                   float* __restrict__ scale, float* __restrict__ running) {
  float m = 0.0f;
  for (int i = threadIdx.x; i < n_partial; i += 256) m = fmaxf(m, __ldcg(partial_at(q, ldq, per_row, per_row_inv, first, i)));
  m = warp_max(m);
  __shared__ float smax[8];
  if ((threadIdx.x & 31) == 0) smax[threadIdx.x >> 5] = m;
  __syncthreads();
  m = smax[threadIdx.x & 7];
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  float s = __fdiv_rn(m, 127.0f);
  if (!(s > 0.0f)) s = 1.0f;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    if (scale) *scale = s;
    if (running) *running = fmaxf(*running, m);
  }
  return s;
}
__global__ void __launch_bounds__(256) partials_to_scale_kernel(uint8_t* q, int64_t ldq, uint32_t per_row, uint64_t per_row_inv, int n_partial,
                                                                float* __restrict__ scale, float* __restrict__ running) {
  grid_dependency_wait();
  grid_dependency_release();
  scale_of_partials(q, ldq, per_row, per_row_inv, 0, n_partial, scale, running);
}
// V pieces per thread
template <typename T, int V>
__global__ void __launch_bounds__(256) act_quant_dynamic_kernel(const T* x, int64_t M, int64_t K, int64_t ldx, uint64_t per_row_inv, int n_partial,
                                                                float* __restrict__ scale, float* __restrict__ running, uint8_t* q, int64_t ldq) {
  grid_dependency_wait();
  grid_dependency_release();
  const uint32_t per_row = static_cast<uint32_t>(K / 8);
  const int64_t total = M * (K / 8);
  const int64_t first = part_first(total, gridDim.x, 256 * V, blockIdx.x), last = part_first(total, gridDim.x, 256 * V, blockIdx.x + 1);
  float v[V][8];
  uint8_t* dst[V];
#pragma unroll
  for (int k = 0; k < V; ++k) {
    const uint32_t piece = static_cast<uint32_t>(first) + threadIdx.x + 256u * k, row = row_of(piece, per_row_inv);
    const int64_t col = static_cast<int64_t>(piece - row * per_row) * 8;
    dst[k] = piece < last ? q + row * ldq + col : nullptr;
    if (dst[k]) Load8<T>::load(x + row * ldx + col, v[k]);
  }
  const float inv = __fdiv_rn(1.0f, scale_of_partials(q, ldq, per_row, per_row_inv, first, n_partial, scale, running));
#pragma unroll
  for (int k = 0; k < V; ++k)
    if (dst[k]) *reinterpret_cast<uint2*>(dst[k]) = quantize_pack8(v[k], inv, 0.0f, -127.0f, 127.0f);
}

// Quantizer behind a producer that has left the largest magnitude in *absmax: s = absmax / 127 (1 for an empty range), which thread 0 of
// CTA 0 leaves in *scale and folds into *running.  16 elements per thread, K % 16 == 0, contiguous.  1024 x 1152 f32: 2.9 us, with a pass
// of its own for the range 6.4; 1024 x 4608: 4.9 and 10.7.
__global__ void __launch_bounds__(256) act_quant_absmax_kernel(const float* x, int64_t pieces, const float* absmax,
                                                               float* __restrict__ scale, float* __restrict__ running, uint8_t* __restrict__ q) {
  grid_dependency_wait();
  grid_dependency_release();
  const int64_t idx = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  float a[8], b[8];
  if (idx < pieces) {
    Load8<float>::load(x + idx * 16, a);
    Load8<float>::load(x + idx * 16 + 8, b);
  }
  const float m = *absmax;
  float s = __fdiv_rn(m, 127.0f);
  if (!(s > 0.0f)) s = 1.0f;
  if (idx == 0) {
    *scale = s;
    *running = fmaxf(*running, m);
  }
  if (idx < pieces) {
    const float inv = __fdiv_rn(1.0f, s);
    const uint2 lo = quantize_pack8(a, inv, 0.0f, -127.0f, 127.0f), hi = quantize_pack8(b, inv, 0.0f, -127.0f, 127.0f);
    *reinterpret_cast<uint4*>(q + idx * 16) = make_uint4(lo.x, lo.y, hi.x, hi.y);
  }
}

// scale[i] = absmax[i] / 127 (1 if the range is empty).
__global__ void absmax_to_scale_kernel(const float* __restrict__ absmax, float* __restrict__ scale, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float s = __fdiv_rn(absmax[i], 127.0f);
  scale[i] = s > 0.0f ? s : 1.0f;
}

// ----------------------------------------------------------------------------- channel-wise weight quantizer
// One CTA per output row: abs-max over K, then codes and their sum.
__global__ void __launch_bounds__(256) weight_quant_kernel(const float* __restrict__ w, int64_t K,
                                                           int8_t* __restrict__ q, float* __restrict__ w_scale,
                                                           int32_t* __restrict__ w_colsum, float top) {
  const int64_t n = blockIdx.x;
  const float* row = w + n * K;
  __shared__ float sm[8];
  __shared__ int si[8];
  float m = 0.0f;
  for (int64_t k = threadIdx.x * 4; k < K; k += blockDim.x * 4) {
    const float4 v = *reinterpret_cast<const float4*>(row + k);
    m = fmaxf(fmaxf(m, fmaxf(fabsf(v.x), fabsf(v.y))), fmaxf(fabsf(v.z), fabsf(v.w)));
  }
  m = warp_max(m);
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = m;
  __syncthreads();
  m = 0.0f;
  for (int i = 0; i < (blockDim.x >> 5); ++i) m = fmaxf(m, sm[i]);
  float s = __fdiv_rn(m, top);
  if (!(s > 0.0f)) s = 1.0f;
  const float inv = __fdiv_rn(1.0f, s);
  int sum = 0;
  for (int64_t k = threadIdx.x * 4; k < K; k += blockDim.x * 4) {
    const float4 v = *reinterpret_cast<const float4*>(row + k);
    const int c0 = __float2int_rn(quantize_code(v.x, inv, 0.0f, -top, top));
    const int c1 = __float2int_rn(quantize_code(v.y, inv, 0.0f, -top, top));
    const int c2 = __float2int_rn(quantize_code(v.z, inv, 0.0f, -top, top));
    const int c3 = __float2int_rn(quantize_code(v.w, inv, 0.0f, -top, top));
    sum += c0 + c1 + c2 + c3;
    const uint32_t packed = (c0 & 0xFF) | ((c1 & 0xFF) << 8) | ((c2 & 0xFF) << 16) | (static_cast<uint32_t>(c3 & 0xFF) << 24);
    *reinterpret_cast<uint32_t*>(q + n * K + k) = packed;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if ((threadIdx.x & 31) == 0) si[threadIdx.x >> 5] = sum;
  __syncthreads();
  if (threadIdx.x == 0) {
    int t = 0;
    for (int i = 0; i < (blockDim.x >> 5); ++i) t += si[i];
    w_scale[n] = s;
    w_colsum[n] = t;
  }
}

// ----------------------------------------------------------------------------- LayerNorm + modulate (+ quantize)
// A CTA owns a contiguous range of rows; its 8 warps take the rows in turn, one warp per row, the row in
// registers (NV vectors of 8 per lane), statistics two-pass in f32.  While a warp works on one row the next
// row's loads are already in flight.  The kernel is bound by instruction issue, so everything that does not
// depend on the row is done once per CTA: for the (at most two) samples its range touches, the per-column
// factors  mul = (1 + scale) / s_out  and  add = shift / s_out  (s_out = 1 unless the output is quantized) are
// staged in shared memory, laid out so that a lane's 16-byte reads are conflict-free.  Per element that leaves
// y / s_out = (x - mean) * (rstd * mul) + add: one multiply and one fused multiply-add.  A row of a third
// sample (only when a sample has fewer rows than a CTA's minimum range) computes its factors from global memory.
template <int NV>
__device__ __forceinline__ void ln_load_row(const __nv_bfloat16* __restrict__ xr, int nvec, int lane, uint4 (&raw)[NV]) {
#pragma unroll
  for (int j = 0; j < NV; ++j) {
    const int vi = lane + 32 * j;
    if (vi < nvec) raw[j] = *reinterpret_cast<const uint4*>(xr + vi * 8);
  }
}

template <int NV, bool MAX, bool EARLY>   // MAX: f32 output whose largest magnitude goes to *absmax; EARLY: see ln_modulate_q8_kernel
__global__ void __launch_bounds__(256) ln_modulate_kernel(const __nv_bfloat16* __restrict__ x, int M, int D, int T,
                                                          float eps, const float* __restrict__ shift,
                                                          const float* __restrict__ scale, int64_t ld_mod,
                                                          void* __restrict__ out, int out_dtype, QuantArgs qa,
                                                          int rows_per_cta, float* __restrict__ absmax) {
  extern __shared__ float4 s_par[];  // [2 samples][mul, add][NV][2 halves][32 lanes]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const int row_begin = blockIdx.x * rows_per_cta;
  const int row_end = row_begin + rows_per_cta < M ? row_begin + rows_per_cta : M;
  if (row_begin >= M) return;
  const int nvec = D >> 3;
  int row = row_begin + warp;
  uint4 raw[NV], raw_next[NV];
  if constexpr (!EARLY) {
    grid_dependency_wait();
    grid_dependency_release();
    if (row < row_end) ln_load_row<NV>(x + static_cast<int64_t>(row) * D, nvec, lane, raw);
  }
  float inv = 1.0f;
  if (out_dtype == QDIT_I8) inv = __fdiv_rn(1.0f, qa.scale_dev ? __ldg(qa.scale_dev) : qa.scale);
  const int b0 = row_begin / T;
  for (int s = 0; s < 2; ++s) {
    if (static_cast<int64_t>(b0 + s) * T >= row_end) break;
    const float* gs = shift + (b0 + s) * ld_mod;
    const float* gc = scale + (b0 + s) * ld_mod;
    for (int i = threadIdx.x; i < NV * 64; i += blockDim.x) {
      const int l = i & 31, h = (i >> 5) & 1, j = i >> 6;
      const int vi = l + 32 * j;
      if (vi < nvec) {
        const float4 c4 = *reinterpret_cast<const float4*>(gc + vi * 8 + 4 * h);
        const float4 h4 = *reinterpret_cast<const float4*>(gs + vi * 8 + 4 * h);
        s_par[(s * 2 + 0) * NV * 64 + i] = make_float4((1.0f + c4.x) * inv, (1.0f + c4.y) * inv, (1.0f + c4.z) * inv, (1.0f + c4.w) * inv);
        s_par[(s * 2 + 1) * NV * 64 + i] = make_float4(h4.x * inv, h4.y * inv, h4.z * inv, h4.w * inv);
      }
    }
  }
  if constexpr (EARLY) {
    grid_dependency_wait();
    grid_dependency_release();
    if (row < row_end) ln_load_row<NV>(x + static_cast<int64_t>(row) * D, nvec, lane, raw);
  }
  __syncthreads();
  const float inv_d = 1.0f / static_cast<float>(D);
  const int64_t second = static_cast<int64_t>(b0 + 1) * T;  // first row of the second staged sample
  [[maybe_unused]] float top = 0.0f;
  for (; row < row_end; row += nwarps) {
    const int next = row + nwarps;
    if (next < row_end) ln_load_row<NV>(x + static_cast<int64_t>(next) * D, nvec, lane, raw_next);
    float v[NV][8];
    float sum = 0.0f;
#pragma unroll
    for (int j = 0; j < NV; ++j) {
      if (lane + 32 * j < nvec) {
        unpack_bf16x2(raw[j].x, v[j][0], v[j][1]);
        unpack_bf16x2(raw[j].y, v[j][2], v[j][3]);
        unpack_bf16x2(raw[j].z, v[j][4], v[j][5]);
        unpack_bf16x2(raw[j].w, v[j][6], v[j][7]);
#pragma unroll
        for (int i = 0; i < 8; ++i) sum += v[j][i];
      }
    }
    const float mean = warp_sum(sum) * inv_d;
    float ssq = 0.0f;
#pragma unroll
    for (int j = 0; j < NV; ++j) {
      if (lane + 32 * j < nvec) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          v[j][i] -= mean;
          ssq = fmaf(v[j][i], v[j][i], ssq);
        }
      }
    }
    const float rstd = rsqrtf(warp_sum(ssq) * inv_d + eps);
    const int sidx = row < second ? 0 : (row - second < T ? 1 : 2);
    const float4* pm = s_par + (sidx * 2 + 0) * NV * 64 + lane;
    const float4* pa = s_par + (sidx * 2 + 1) * NV * 64 + lane;
#pragma unroll
    for (int j = 0; j < NV; ++j) {
      const int vi = lane + 32 * j;
      if (vi < nvec) {
        float mul[8], add[8], y[8];
        if (sidx < 2) {
          const float4 m0 = pm[j * 64], m1 = pm[j * 64 + 32], a0 = pa[j * 64], a1 = pa[j * 64 + 32];
          mul[0] = m0.x; mul[1] = m0.y; mul[2] = m0.z; mul[3] = m0.w; mul[4] = m1.x; mul[5] = m1.y; mul[6] = m1.z; mul[7] = m1.w;
          add[0] = a0.x; add[1] = a0.y; add[2] = a0.z; add[3] = a0.w; add[4] = a1.x; add[5] = a1.y; add[6] = a1.z; add[7] = a1.w;
        } else {
          const int b = row / T;
          Load8<float>::load(scale + b * ld_mod + vi * 8, mul);
          Load8<float>::load(shift + b * ld_mod + vi * 8, add);
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            mul[i] = (1.0f + mul[i]) * inv;
            add[i] *= inv;
          }
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) y[i] = fmaf(v[j][i], rstd * mul[i], add[i]);
        const int64_t o = static_cast<int64_t>(row) * D + vi * 8;
        if (out_dtype == QDIT_I8) {
          *reinterpret_cast<uint2*>(static_cast<uint8_t*>(out) + o) = quantize_pack8_scaled(y, qa.zp, qa.qmin, qa.qmax);
        } else if (out_dtype == QDIT_BF16) {
          *reinterpret_cast<uint4*>(static_cast<__nv_bfloat16*>(out) + o) = pack_bf16x8(y);
        } else {
          if constexpr (MAX) {
#pragma unroll
            for (int i = 0; i < 8; ++i) top = fmaxf(top, fabsf(y[i]));
          }
          float* of = static_cast<float*>(out) + o;
          *reinterpret_cast<float4*>(of) = make_float4(y[0], y[1], y[2], y[3]);
          *reinterpret_cast<float4*>(of + 4) = make_float4(y[4], y[5], y[6], y[7]);
        }
      }
    }
#pragma unroll
    for (int j = 0; j < NV; ++j) raw[j] = raw_next[j];
  }
  if constexpr (MAX) publish_absmax(absmax, top);
}

// The same operation for the shape the network's blocks use: 8-bit output and D = 128 * NV4.  A lane owns NV4
// groups of 4 consecutive columns (group lane + 32 j), so all 32 lanes are busy for every group (D = 1152 has 4.5
// groups of 8 per lane, which leaves half a warp idle for a fifth of the work), and the f32 arithmetic runs on
// the two-wide instructions (add / mul / fma on a pair of floats: same rounding per element as the scalar forms).
// Together that is less than half of the general kernel's instructions per row.  Values are identical to the
// general kernel's except for the summation order of the two statistics.  A CTA's row range must lie within two
// samples (rows_per_cta <= T).
__device__ __forceinline__ float2 f2(float a, float b) { return make_float2(a, b); }

// 28 warps per SM (two CTAs of 14): at the 8192 rows of the 256-token workload a warp then has two rows; with 24 it had 2.3,
// that is three turns.  The next row is fetched into the registers of the current one as soon as that one is widened.
constexpr int LNQ_WARPS = 14;
template <int NV4, bool EARLY>
__global__ void __launch_bounds__(LNQ_WARPS * 32, 2) ln_modulate_q8_kernel(const __nv_bfloat16* __restrict__ x, int M, int T, float eps,
                                                                const float* __restrict__ shift,
                                                                const float* __restrict__ scale, int64_t ld_mod,
                                                                uint8_t* __restrict__ out, QuantArgs qa, int rows_per_cta) {
  constexpr int D = NV4 * 128, D4 = D / 4;
  extern __shared__ float4 s_par[];  // [2 samples][mul, add][D / 4]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int row_begin = blockIdx.x * rows_per_cta;
  const int row_end = row_begin + rows_per_cta < M ? row_begin + rows_per_cta : M;
  if (row_begin >= M) return;
  int row = row_begin + warp;
  uint2 raw[NV4];
  auto load_row = [&]() {
    if (row < row_end) {
      const uint2* xr = reinterpret_cast<const uint2*>(x + static_cast<int64_t>(row) * D) + lane;
#pragma unroll
      for (int j = 0; j < NV4; ++j) raw[j] = xr[32 * j];
    }
  };
  // EARLY: the modulation and the scale were written two launches ago or earlier and are staged while the previous kernel, which writes
  // x, still runs.  (Not a run-time choice: rows loaded in a branch are waited for behind it, and the two latencies add up: 1024 x 1152 with f32
  // output 3.5 us by itself instead of 3.2.)
  if constexpr (!EARLY) {
    grid_dependency_wait();
    grid_dependency_release();
    load_row();
  }
  const float inv = __fdiv_rn(1.0f, device_value(qa.scale_dev, qa.scale));
  const int b0 = row_begin / T;
  for (int s = 0; s < 2; ++s) {
    if (static_cast<int64_t>(b0 + s) * T >= row_end) break;
    const float4* gs = reinterpret_cast<const float4*>(shift + (b0 + s) * ld_mod);
    const float4* gc = reinterpret_cast<const float4*>(scale + (b0 + s) * ld_mod);
    for (int i = threadIdx.x; i < D4; i += LNQ_WARPS * 32) {
      const float4 c4 = gc[i], h4 = gs[i];
      s_par[(s * 2 + 0) * D4 + i] = make_float4((1.0f + c4.x) * inv, (1.0f + c4.y) * inv, (1.0f + c4.z) * inv, (1.0f + c4.w) * inv);
      s_par[(s * 2 + 1) * D4 + i] = make_float4(h4.x * inv, h4.y * inv, h4.z * inv, h4.w * inv);
    }
  }
  if constexpr (EARLY) {
    grid_dependency_wait();
    grid_dependency_release();
    load_row();
  }
  __syncthreads();
  constexpr float inv_d = 1.0f / static_cast<float>(D);
  const int second = (b0 + 1) * T;  // first row of the second staged sample
  const float lo_f = qa.qmin - qa.zp, hi_f = qa.qmax - qa.zp;
  const uint32_t z4 = (static_cast<uint32_t>(static_cast<int>(qa.zp)) & 0xFFu) * 0x01010101u;
  const float2 magic = f2(12582912.0f, 12582912.0f);
  for (; row < row_end; row += LNQ_WARPS) {
    float2 v[NV4][2];
    float2 s0 = f2(0.0f, 0.0f), s1 = f2(0.0f, 0.0f);
#pragma unroll
    for (int j = 0; j < NV4; ++j) {
      v[j][0] = f2(__uint_as_float(raw[j].x << 16), __uint_as_float(raw[j].x & 0xFFFF0000u));
      v[j][1] = f2(__uint_as_float(raw[j].y << 16), __uint_as_float(raw[j].y & 0xFFFF0000u));
      s0 = __fadd2_rn(s0, v[j][0]);
      s1 = __fadd2_rn(s1, v[j][1]);
    }
    const int next = row + LNQ_WARPS;
    if (next < row_end) {
      const uint2* xr = reinterpret_cast<const uint2*>(x + static_cast<int64_t>(next) * D) + lane;
#pragma unroll
      for (int j = 0; j < NV4; ++j) raw[j] = xr[32 * j];
    }
    const float mean = warp_sum((s0.x + s0.y) + (s1.x + s1.y)) * inv_d;
    const float2 nmean = f2(-mean, -mean);
    float2 q0 = f2(0.0f, 0.0f), q1 = f2(0.0f, 0.0f);
#pragma unroll
    for (int j = 0; j < NV4; ++j) {
      v[j][0] = __fadd2_rn(v[j][0], nmean);
      v[j][1] = __fadd2_rn(v[j][1], nmean);
      q0 = __ffma2_rn(v[j][0], v[j][0], q0);
      q1 = __ffma2_rn(v[j][1], v[j][1], q1);
    }
    const float rstd = rsqrtf(warp_sum((q0.x + q0.y) + (q1.x + q1.y)) * inv_d + eps);
    const float2 r2 = f2(rstd, rstd);
    const float4* pm = s_par + (row < second ? 0 : 2) * D4 + lane;
    const float4* pa = pm + D4;
    uint32_t* orow = reinterpret_cast<uint32_t*>(out + static_cast<int64_t>(row) * D) + lane;
#pragma unroll
    for (int j = 0; j < NV4; ++j) {
      const float4 m4 = pm[32 * j], a4 = pa[32 * j];
      // y / s_out = (x - mean) * (rstd * mul) + add, then Eq. 1's clip and round on the scaled value
      float2 y0 = __ffma2_rn(v[j][0], __fmul2_rn(r2, f2(m4.x, m4.y)), f2(a4.x, a4.y));
      float2 y1 = __ffma2_rn(v[j][1], __fmul2_rn(r2, f2(m4.z, m4.w)), f2(a4.z, a4.w));
      y0 = __fadd2_rn(f2(fminf(fmaxf(y0.x, lo_f), hi_f), fminf(fmaxf(y0.y, lo_f), hi_f)), magic);
      y1 = __fadd2_rn(f2(fminf(fmaxf(y1.x, lo_f), hi_f), fminf(fmaxf(y1.y, lo_f), hi_f)), magic);
      uint32_t w = __byte_perm(__byte_perm(__float_as_uint(y0.x), __float_as_uint(y0.y), 0x0040),
                               __byte_perm(__float_as_uint(y1.x), __float_as_uint(y1.y), 0x0040), 0x5410);
      if (z4 != 0u) w = __vadd4(w, z4);  // code + z stays inside a byte
      orow[32 * j] = w;
    }
  }
}

template <int NV4>
void launch_ln_q8(qdit_ctx* ctx, const void* x, int64_t M, const float* shift, const float* scale, int64_t ld_mod,
                  int64_t T, float eps, void* out, QuantArgs qa, int64_t rows, bool early) {
  const unsigned grid = static_cast<unsigned>((M + rows - 1) / rows);
  qdit_launch_overlapped(ctx, early ? ln_modulate_q8_kernel<NV4, true> : ln_modulate_q8_kernel<NV4, false>, dim3(grid), dim3(LNQ_WARPS * 32), static_cast<size_t>(NV4) * 128 * 16,
                         static_cast<const __nv_bfloat16*>(x), static_cast<int>(M), static_cast<int>(T), eps, shift, scale,
                         ld_mod, static_cast<uint8_t*>(out), qa, static_cast<int>(rows));
}

// Row range per CTA: `per_sm` CTAs per SM, at least eight rows, at most what keeps a range within two samples.
int64_t ln_rows_per_cta(const qdit_ctx* ctx, int64_t M, int64_t T, int per_sm) {
  const int64_t ctas = per_sm * static_cast<int64_t>(ctx->num_sms);
  int64_t rows = (M + ctas - 1) / ctas;
  if (rows < 8) rows = 8;
  if (rows > T) rows = T;
  return rows;
}

template <int NV>
void launch_ln(qdit_ctx* ctx, const void* x, int64_t M, int D, int64_t T, float eps, const float* shift,
               const float* scale, int64_t ld_mod, void* out, int out_dtype, QuantArgs qa, bool early, float* absmax) {
  const int64_t rows = ln_rows_per_cta(ctx, M, T, 2);
  const unsigned grid = static_cast<unsigned>((M + rows - 1) / rows);
  const auto kernel = absmax ? (early ? ln_modulate_kernel<NV, true, true> : ln_modulate_kernel<NV, true, false>)
                             : (early ? ln_modulate_kernel<NV, false, true> : ln_modulate_kernel<NV, false, false>);
  qdit_launch_overlapped(ctx, kernel, dim3(grid), dim3(256), static_cast<size_t>(NV) * 4096,
                         static_cast<const __nv_bfloat16*>(x), static_cast<int>(M), D, static_cast<int>(T), eps, shift, scale,
                         ld_mod, out, out_dtype, qa, static_cast<int>(rows), absmax);
}

}  // namespace

namespace {
template <typename... KArgs, typename... Args>
cudaError_t launch_act_quant(qdit_ctx* ctx, unsigned early_ctas, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, Args&&... args) {
  if (grid.x <= early_ctas) return qdit_launch_overlapped(ctx, kernel, grid, block, smem, args...);
  kernel<<<grid, block, smem, ctx->stream>>>(static_cast<KArgs>(args)...);
  return cudaGetLastError();
}

template <typename T>
int32_t quant_dynamic(qdit_ctx* ctx, const T* x, int64_t M, int64_t K, int64_t ldx, float* scale, float* running, uint8_t* q, int64_t ldq) {
  const int64_t total = M * (K / 8);
  const uint64_t per_row_inv = inverse_of(K / 8);
  ProfScope prof(ctx, QDIT_PROF_ACT_QUANT, static_cast<double>(M) * K * (sizeof(T) + 1.0));
  if (total <= DYN_PIECES) {
    // one piece per thread for up to 512 parts; then two, four, eight.  With more parts than SMs one larger CTA per SM forms the
    // partials (512 x 1152, bf16: 4.0 us, with one CTA per part 4.4; two pieces per thread there 4.6)
    const int v = total <= 512 * 256 ? 1 : total <= 300 * 512 ? 2 : total <= 300 * 1024 ? 4 : 8;
    const int parts = static_cast<int>((total + 256 * v - 1) / (256 * v));
    const int n_partial = parts < ctx->num_sms ? parts : ctx->num_sms < DYN_PARTIALS ? ctx->num_sms : DYN_PARTIALS;
    const int threads = n_partial == parts ? 256 : v == 1 ? 512 : 1024;
    const auto quantize = v == 1 ? act_quant_dynamic_kernel<T, 1> : v == 2 ? act_quant_dynamic_kernel<T, 2> : v == 4 ? act_quant_dynamic_kernel<T, 4> : act_quant_dynamic_kernel<T, 8>;
    QDIT_CUDA_CHECK(ctx, qdit_launch_overlapped(ctx, threads == 256 ? absmax_partial_kernel<T, 256> : threads == 512 ? absmax_partial_kernel<T, 512> : absmax_partial_kernel<T, 1024>, dim3(n_partial), dim3(threads), 0, x, M, K,
                                                ldx, q, ldq, per_row_inv, parts, 256 * v));
    QDIT_TRY(qdit_after_launch(ctx, "absmax_partial_kernel"));
    QDIT_CUDA_CHECK(ctx, qdit_launch_overlapped(ctx, quantize, dim3(parts), dim3(256), 0, x, M, K, ldx, per_row_inv, n_partial, scale, running, q, ldq));
    return qdit_after_launch(ctx, "act_quant_dynamic_kernel");
  }
  const int n_partial = ctx->num_sms * 8;   // fewer than the pieces of a tensor that comes here
  QDIT_CUDA_CHECK(ctx, qdit_launch_overlapped(ctx, absmax_partial_kernel<T, 256>, dim3(n_partial), dim3(256), 0, x, M, K, ldx, q, ldq, per_row_inv, 1, 0));
  QDIT_TRY(qdit_after_launch(ctx, "absmax_partial_kernel"));
  QDIT_CUDA_CHECK(ctx, qdit_launch_overlapped(ctx, partials_to_scale_kernel, dim3(1), dim3(256), 0, q, ldq, static_cast<uint32_t>(K / 8), per_row_inv, n_partial, scale, running));
  QDIT_TRY(qdit_after_launch(ctx, "partials_to_scale_kernel"));
  const QuantArgs qa = make_quant_args(qdit_qparams{1.0f, 0, -127, 127}, scale);
  const int64_t threads = M * ((K + 15) / 16);
  // (the launch in front is one CTA: nothing to be packed beside)
  QDIT_CUDA_CHECK(ctx, launch_act_quant(ctx, RELEASE_CTAS, act_quant_kernel<T>, dim3(static_cast<unsigned>((threads + 255) / 256)), dim3(256), 0, x, M, K, ldx, qa,
                                              q, ldq));
  return qdit_after_launch(ctx, "act_quant_kernel");
}

// The rows stay in registers where enough warps fit beside them: 2 or 5 pieces per lane (us, row read twice / kept, bf16: 65536 x 384
// 24.8 / 16.2, 5000 x 1152 5.0 / 4.3, 65536 x 1152 45.5 / 38.7; f32 62.8 / 54.8), and 18 of bf16 for few long rows, where only the latency
// counts (64 x 4608 4.8 / 3.5; 5000 x 4608 12.1 / 14.8, and 5000 x 1536 5.5 / 9.8 with two thirds of the pieces missing).
template <typename T>
int32_t quant_token(qdit_ctx* ctx, const T* x, int64_t M, int64_t K, int64_t ldx, float* scales, uint8_t* q, int64_t ldq) {
  constexpr bool NARROW = sizeof(T) == 2;
  const auto kernel = K <= 512 ? act_quant_token_kernel<T, 2> : K <= 1280 ? act_quant_token_kernel<T, 5> : NARROW && K > 2304 && K <= 4608 && M <= 512 ? act_quant_token_kernel<T, NARROW ? 18 : 0>
                                                                                                        : act_quant_token_kernel<T, 0>;
  QDIT_CUDA_CHECK(ctx, launch_act_quant(ctx, EARLY_TOKEN_CTAS, kernel, dim3(static_cast<unsigned>((M + 7) / 8)), dim3(256), 0, x, M, K, ldx, scales, q, ldq));
  return qdit_after_launch(ctx, "act_quant_token_kernel");
}
}  // namespace

int32_t launch_quant_dynamic(qdit_ctx* ctx, const void* x, int x_dtype, int64_t M, int64_t K, int64_t ldx, float* scale,
                             float* running, void* q, int64_t ldq) {
  if (M == 0 || K == 0) return QDIT_OK;
  if (x_dtype == QDIT_BF16) return quant_dynamic(ctx, static_cast<const __nv_bfloat16*>(x), M, K, ldx, scale, running, static_cast<uint8_t*>(q), ldq);
  return quant_dynamic(ctx, static_cast<const float*>(x), M, K, ldx, scale, running, static_cast<uint8_t*>(q), ldq);
}

int32_t launch_quant_absmax(qdit_ctx* ctx, const float* x, int64_t M, int64_t K, const float* absmax, float* scale, float* running, void* q) {
  const int64_t pieces = M * K / 16;
  if (pieces == 0) return QDIT_OK;
  ProfScope prof(ctx, QDIT_PROF_ACT_QUANT, static_cast<double>(M) * K * 5.0);
  QDIT_CUDA_CHECK(ctx, launch_act_quant(ctx, EARLY_CTAS, act_quant_absmax_kernel, dim3(static_cast<unsigned>((pieces + 255) / 256)), dim3(256), 0, x, pieces, absmax,
                                        scale, running, static_cast<uint8_t*>(q)));
  return qdit_after_launch(ctx, "act_quant_absmax_kernel");
}

int32_t launch_absmax_to_scale(qdit_ctx* ctx, const float* absmax_dev, float* scale_dev, int n) {
  if (n <= 0) return QDIT_OK;
  absmax_to_scale_kernel<<<(n + 127) / 128, 128, 0, ctx->stream>>>(absmax_dev, scale_dev, n);
  return qdit_after_launch(ctx, "absmax_to_scale_kernel");
}

int32_t qdit_quantize_act_dev(qdit_ctx* ctx, const float* x, int64_t M, int64_t K, qdit_qparams qp,
                              const float* scale_dev, uint8_t* q) {
  if (M == 0 || K == 0) return QDIT_OK;
  const QuantArgs qa = make_quant_args(qp, scale_dev);
  const int64_t threads = M * ((K + 15) / 16);
  QDIT_CUDA_CHECK(ctx, launch_act_quant(ctx, EARLY_CTAS, act_quant_kernel<float>, dim3(static_cast<unsigned>((threads + 255) / 256)), dim3(256), 0, x, M, K, K, qa, q, K));
  return qdit_after_launch(ctx, "act_quant_kernel");
}

extern "C" {

int32_t qdit_quantize_act(qdit_ctx* ctx, const void* x, int x_dtype, int64_t M, int64_t K, int64_t ldx, int mode,
                          const qdit_qparams* qp, float* dyn_scale, void* q, int64_t ldq) {
  if (!ctx) return QDIT_ERR_INVALID_ARG;
  if (M < 0 || K < 0) return qdit_fail(ctx, QDIT_ERR_SHAPE, "negative size");
  if (M == 0 || K == 0) return QDIT_OK;
  if (!x || !q) return qdit_fail(ctx, QDIT_ERR_INVALID_ARG, "x or q is NULL");
  if (x_dtype != QDIT_BF16 && x_dtype != QDIT_F32) return qdit_fail(ctx, QDIT_ERR_INVALID_ARG, "x_dtype must be bf16 or f32");
  if (K % 8 != 0) return qdit_fail(ctx, QDIT_ERR_SHAPE, "K = %lld must be a multiple of 8", static_cast<long long>(K));
  if (ldx < K || ldq < K) return qdit_fail(ctx, QDIT_ERR_SHAPE, "leading dimension smaller than K");
  const int64_t esz = x_dtype == QDIT_BF16 ? 2 : 4;
  if (!aligned16(x) || (ldx * esz) % 16 != 0) return qdit_fail(ctx, QDIT_ERR_ALIGN, "x must be 16-byte aligned (base and row pitch)");
  if ((reinterpret_cast<uintptr_t>(q) & 7u) || ldq % 8 != 0) return qdit_fail(ctx, QDIT_ERR_ALIGN, "q must be 8-byte aligned (base and row pitch)");
  QuantArgs qa;
  if (mode == QDIT_QUANT_STATIC) {
    QDIT_TRY(qdit_check_qparams(ctx, qp, false));
    qa = make_quant_args(*qp, nullptr);
  } else if (mode == QDIT_QUANT_DYNAMIC_TOKEN) {
    if (!dyn_scale) return qdit_fail(ctx, QDIT_ERR_INVALID_ARG, "per-token mode needs dyn_scale [M]");
    if (x_dtype == QDIT_BF16) return quant_token(ctx, static_cast<const __nv_bfloat16*>(x), M, K, ldx, dyn_scale, static_cast<uint8_t*>(q), ldq);
    return quant_token(ctx, static_cast<const float*>(x), M, K, ldx, dyn_scale, static_cast<uint8_t*>(q), ldq);
  } else if (mode == QDIT_QUANT_DYNAMIC) {
    if (!dyn_scale) return qdit_fail(ctx, QDIT_ERR_INVALID_ARG, "dynamic mode needs dyn_scale");
    return launch_quant_dynamic(ctx, x, x_dtype, M, K, ldx, dyn_scale, nullptr, q, ldq);
  } else {
    return qdit_fail(ctx, QDIT_ERR_INVALID_ARG, "unknown quantizer mode %d", mode);
  }
  const int64_t threads = M * ((K + 15) / 16);
  const unsigned grid = static_cast<unsigned>((threads + 255) / 256);
  ProfScope prof(ctx, QDIT_PROF_ACT_QUANT, static_cast<double>(M) * K * (esz + 1.0));
  if (x_dtype == QDIT_BF16)
    QDIT_CUDA_CHECK(ctx, launch_act_quant(ctx, EARLY_CTAS, act_quant_kernel<__nv_bfloat16>, dim3(grid), dim3(256), 0, static_cast<const __nv_bfloat16*>(x), M, K, ldx, qa,
                                                                   static_cast<uint8_t*>(q), ldq));
  else
    QDIT_CUDA_CHECK(ctx, launch_act_quant(ctx, EARLY_CTAS, act_quant_kernel<float>, dim3(grid), dim3(256), 0, static_cast<const float*>(x), M, K, ldx, qa,
                                                           static_cast<uint8_t*>(q), ldq));
  return qdit_after_launch(ctx, "act_quant_kernel");
}

int32_t qdit_quantize_weight_bits(qdit_ctx* ctx, const float* w, int64_t N, int64_t K, int bits, void* q, float* w_scale,
                             int32_t* w_colsum) {
  if (!ctx) return QDIT_ERR_INVALID_ARG;
  if (bits < 2 || bits > 8) return qdit_fail(ctx, QDIT_ERR_INVALID_ARG, "bits = %d outside 2..8", bits);
  if (N < 0 || K < 0) return qdit_fail(ctx, QDIT_ERR_SHAPE, "negative size");
  if (N == 0 || K == 0) return QDIT_OK;
  if (!w || !q || !w_scale || !w_colsum) return qdit_fail(ctx, QDIT_ERR_INVALID_ARG, "NULL argument");
  if (K % 4 != 0) return qdit_fail(ctx, QDIT_ERR_SHAPE, "K must be a multiple of 4");
  if (!aligned16(w) || (reinterpret_cast<uintptr_t>(q) & 3u)) return qdit_fail(ctx, QDIT_ERR_ALIGN, "w must be 16-byte, q 4-byte aligned");
  weight_quant_kernel<<<static_cast<unsigned>(N), 256, 0, ctx->stream>>>(w, K, static_cast<int8_t*>(q), w_scale, w_colsum,
                                                                         static_cast<float>((1 << (bits - 1)) - 1));
  return qdit_after_launch(ctx, "weight_quant_kernel");
}

int32_t qdit_quantize_weight(qdit_ctx* ctx, const float* w, int64_t N, int64_t K, void* q, float* w_scale,
                             int32_t* w_colsum) {
  return qdit_quantize_weight_bits(ctx, w, N, K, 8, q, w_scale, w_colsum);
}

int32_t qdit_adaln_modulate(qdit_ctx* ctx, const void* x, int64_t M, int64_t D, int64_t T, float eps,
                            const float* shift, const float* scale, int64_t ld_mod, void* out, int out_dtype,
                            const qdit_qparams* out_qp, const float* out_scale_dev) {
  return qdit_adaln_impl(ctx, x, M, D, T, eps, shift, scale, ld_mod, out, out_dtype, out_qp, out_scale_dev, false, nullptr);
}

}  // extern "C"

int32_t qdit_adaln_impl(qdit_ctx* ctx, const void* x, int64_t M, int64_t D, int64_t T, float eps, const float* shift, const float* scale,
                        int64_t ld_mod, void* out, int out_dtype, const qdit_qparams* out_qp, const float* out_scale_dev, bool early, float* absmax) {
  if (!ctx) return QDIT_ERR_INVALID_ARG;
  if (M < 0 || D <= 0 || T <= 0) return qdit_fail(ctx, QDIT_ERR_SHAPE, "bad sizes");
  if (M > (int64_t(1) << 30) || T > (int64_t(1) << 30)) return qdit_fail(ctx, QDIT_ERR_SHAPE, "M and T must be at most 2^30");
  if (M == 0) return QDIT_OK;
  if (!x || !shift || !scale || !out) return qdit_fail(ctx, QDIT_ERR_INVALID_ARG, "NULL argument");
  if (D % 8 != 0 || D > 2048) return qdit_fail(ctx, QDIT_ERR_SHAPE, "D must be a multiple of 8 and <= 2048");
  if (ld_mod % 4 != 0 || !aligned16(shift) || !aligned16(scale) || !aligned16(x) || !aligned16(out))
    return qdit_fail(ctx, QDIT_ERR_ALIGN, "pointers must be 16-byte aligned and ld_mod a multiple of 4");
  if (out_dtype != QDIT_I8 && out_dtype != QDIT_BF16 && out_dtype != QDIT_F32)
    return qdit_fail(ctx, QDIT_ERR_INVALID_ARG, "bad out_dtype");
  QuantArgs qa{};
  if (out_dtype == QDIT_I8) {
    QDIT_TRY(qdit_check_qparams(ctx, out_qp, out_scale_dev != nullptr));
    qa = make_quant_args(*out_qp, out_scale_dev);
  }
  const int nv = static_cast<int>((D / 8 + 31) / 32);
  const int d = static_cast<int>(D);
  const double out_bytes = out_dtype == QDIT_I8 ? 1.0 : out_dtype == QDIT_BF16 ? 2.0 : 4.0;
  ProfScope prof(ctx, QDIT_PROF_LN_MODULATE, static_cast<double>(M) * D * (2.0 + out_bytes));
  if (out_dtype == QDIT_I8 && D % 128 == 0) {
    // the widths of the DiT family (S 384, B 768, L 1024, XL 1152) with 8-bit output: the two-wide kernel
    const int64_t rows = ln_rows_per_cta(ctx, M, T, 2);
    bool done = true;
    switch (D / 128) {
      case 3: launch_ln_q8<3>(ctx, x, M, shift, scale, ld_mod, T, eps, out, qa, rows, early); break;
      case 6: launch_ln_q8<6>(ctx, x, M, shift, scale, ld_mod, T, eps, out, qa, rows, early); break;
      case 8: launch_ln_q8<8>(ctx, x, M, shift, scale, ld_mod, T, eps, out, qa, rows, early); break;
      case 9: launch_ln_q8<9>(ctx, x, M, shift, scale, ld_mod, T, eps, out, qa, rows, early); break;
      default: done = false; break;
    }
    if (done) return qdit_after_launch(ctx, "ln_modulate_q8_kernel");
  }
  switch (nv) {
    case 1: launch_ln<1>(ctx, x, M, d, T, eps, shift, scale, ld_mod, out, out_dtype, qa, early, absmax); break;
    case 2: launch_ln<2>(ctx, x, M, d, T, eps, shift, scale, ld_mod, out, out_dtype, qa, early, absmax); break;
    case 3: launch_ln<3>(ctx, x, M, d, T, eps, shift, scale, ld_mod, out, out_dtype, qa, early, absmax); break;
    case 4: launch_ln<4>(ctx, x, M, d, T, eps, shift, scale, ld_mod, out, out_dtype, qa, early, absmax); break;
    case 5: launch_ln<5>(ctx, x, M, d, T, eps, shift, scale, ld_mod, out, out_dtype, qa, early, absmax); break;
    case 6: launch_ln<6>(ctx, x, M, d, T, eps, shift, scale, ld_mod, out, out_dtype, qa, early, absmax); break;
    case 7: launch_ln<7>(ctx, x, M, d, T, eps, shift, scale, ld_mod, out, out_dtype, qa, early, absmax); break;
    default: launch_ln<8>(ctx, x, M, d, T, eps, shift, scale, ld_mod, out, out_dtype, qa, early, absmax); break;
  }
  return qdit_after_launch(ctx, "ln_modulate_kernel");
}
