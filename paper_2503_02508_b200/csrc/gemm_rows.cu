// W8A8 / W4A8 linear layer of one to four rows with f32 output (the modulation of one to four images: 193536 channels of 1152).
//
// What bounds it: the weights are read once, from HBM, and each code is used one to four times, so this is a stream of weights with
// a dot product beside it (dp4a: 4 products per lane).  A tile of 128 rows for the tensor core would be one row and 127 of padding,
// fetched in 128-byte pieces of rows 1152 bytes apart, 9 k-blocks one behind the other and an epilogue per tile; here a group
// of eight lanes reads a channel's row in consecutive 128-byte lines, all of it in flight at once (up to 9 x 16 bytes per lane, 32 warps per SM).
//
// 193536 channels of 1152, one row: 35.1 us, 6.4 TB/s (51.2 with the tensor core, 128 x 192 tiles); four rows 45.4, then bound by the
// reads of the activations from shared memory.
//
// Four groups per warp, one channel each; activations in shared memory, read by all groups at one address.  Packed 4-bit codes stay
// in their nibbles: a nibble in the upper half of its byte is 16 times its value as a signed byte, low nibbles are shifted there, the
// activations are dealt out to match (even and odd codes), and the sum is divided by 16, exactly.
#include "gemm_common.cuh"

namespace {

using namespace qgemm;

constexpr int ROWS_THREADS = 256;

template <bool U>
__device__ __forceinline__ int dot4(uint32_t w, uint32_t x, int acc) {   // signed weights, signed or unsigned activations
  int d;
  if (U) asm("dp4a.s32.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(w), "r"(x), "r"(acc));
  else asm("dp4a.s32.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(w), "r"(x), "r"(acc));
  return d;
}

template <int R, bool W4, bool U>
__global__ void __launch_bounds__(ROWS_THREADS, R == 4 ? 3 : 4) few_rows_kernel(const uint8_t* A, const uint8_t* __restrict__ W, const GemmParams p) {
  constexpr int UN = W4 ? 5 : 9;             // pieces of a lane in flight: 1152 codes are 72 pieces of 16 bytes, packed 36
  constexpr int XV = W4 ? 2 : 1;             // 16-byte pieces of activations per piece of weights
  extern __shared__ uint4 xs[];              // [R][XV][pieces]
  const int pieces = p.K / (W4 ? 32 : 16);
  const int lane = threadIdx.x & 31, l = lane & 7;
  const int first = (static_cast<int>(blockIdx.x) * (ROWS_THREADS / 32) + static_cast<int>(threadIdx.x >> 5)) * 4;   // the warp's four channels (N % 8 == 0)
  uint4 w[UN];
  auto fetch = [&](int n, int c0) {
    const uint4* row = reinterpret_cast<const uint4*>(W) + static_cast<int64_t>(n) * pieces;
#pragma unroll
    for (int u = 0; u < UN; ++u) {
      const int c = c0 + 8 * u + l;
      w[u] = c < pieces ? __ldg(row + c) : make_uint4(0u, 0u, 0u, 0u);
    }
  };
  bool fetched = p.early && first < p.N;     // constants may be read before the input is ready
  if (fetched) fetch(first + (lane >> 3), 0);
  grid_dependency_wait();
  grid_dependency_release();
  for (int i = threadIdx.x; i < R * pieces; i += ROWS_THREADS) {
    const int r = i / pieces, c = i - r * pieces;
    const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
    const uint4* src = reinterpret_cast<const uint4*>(A + static_cast<int64_t>(r) * p.K) + c * XV;
    const uint4 a = r < p.M ? src[0] : zero;
    if (W4) {
      const uint4 b = r < p.M ? src[1] : zero;
      xs[(r * 2) * pieces + c] = make_uint4(__byte_perm(a.x, a.y, 0x6420), __byte_perm(a.z, a.w, 0x6420), __byte_perm(b.x, b.y, 0x6420), __byte_perm(b.z, b.w, 0x6420));
      xs[(r * 2 + 1) * pieces + c] = make_uint4(__byte_perm(a.x, a.y, 0x7531), __byte_perm(a.z, a.w, 0x7531), __byte_perm(b.x, b.y, 0x7531), __byte_perm(b.z, b.w, 0x7531));
    } else {
      xs[r * pieces + c] = a;
    }
  }
  const float a_scale = device_value(p.a_scale_dev, p.a_scale);
  __syncthreads();
  for (int nb = first; nb < p.N; nb += static_cast<int>(gridDim.x) * (ROWS_THREADS / 32) * 4) {
    const int n = nb + (lane >> 3);
    const float w_scale = __ldg(p.w_scale + n), bias = __ldg(p.bias + n);
    int acc[R];
#pragma unroll
    for (int r = 0; r < R; ++r) acc[r] = 0;
    for (int c0 = 0; c0 < pieces; c0 += 8 * UN) {
      if (!fetched) fetch(n, c0);
      fetched = false;
#pragma unroll
      for (int u = 0; u < UN; ++u) {
        const int c = c0 + 8 * u + l, cx = c < pieces ? c : 0;   // (past the row's end the weights are zero)
#pragma unroll
        for (int r = 0; r < R; ++r) {
          if (W4) {
            const uint4 e = xs[(r * 2) * pieces + cx], o = xs[(r * 2 + 1) * pieces + cx];
            acc[r] = dot4<U>(w[u].x << 4 & 0xF0F0F0F0u, e.x, acc[r]);
            acc[r] = dot4<U>(w[u].x & 0xF0F0F0F0u, o.x, acc[r]);
            acc[r] = dot4<U>(w[u].y << 4 & 0xF0F0F0F0u, e.y, acc[r]);
            acc[r] = dot4<U>(w[u].y & 0xF0F0F0F0u, o.y, acc[r]);
            acc[r] = dot4<U>(w[u].z << 4 & 0xF0F0F0F0u, e.z, acc[r]);
            acc[r] = dot4<U>(w[u].z & 0xF0F0F0F0u, o.z, acc[r]);
            acc[r] = dot4<U>(w[u].w << 4 & 0xF0F0F0F0u, e.w, acc[r]);
            acc[r] = dot4<U>(w[u].w & 0xF0F0F0F0u, o.w, acc[r]);
          } else {
            const uint4 x = xs[r * pieces + cx];
            acc[r] = dot4<U>(w[u].x, x.x, acc[r]);
            acc[r] = dot4<U>(w[u].y, x.y, acc[r]);
            acc[r] = dot4<U>(w[u].z, x.z, acc[r]);
            acc[r] = dot4<U>(w[u].w, x.w, acc[r]);
          }
        }
      }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
#pragma unroll
      for (int s = 4; s > 0; s >>= 1) acc[r] += __shfl_xor_sync(0xffffffffu, acc[r], s);
    }
    const float sc = __fmul_rn(a_scale, w_scale);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (l == r && r < p.M) {
        int a = W4 ? acc[r] >> 4 : acc[r];
        if (p.a_zp != 0) a -= p.a_zp * __ldg(p.w_colsum + n);
        static_cast<float*>(p.out)[static_cast<int64_t>(r) * p.ldo + n] = __fmaf_rn(static_cast<float>(a), sc, bias);
      }
    }
  }
}

template <int R, bool W4>
int32_t launch_rows(qdit_ctx* ctx, const void* A, const void* W, const GemmParams& p, bool a_unsigned) {
  const int groups = (p.N + ROWS_THREADS / 8 - 1) / (ROWS_THREADS / 8);
  const dim3 grid(groups < (R == 4 ? 3 : 4) * ctx->num_sms ? groups : (R == 4 ? 3 : 4) * ctx->num_sms);
  ProfScope prof(ctx, QDIT_PROF_GEMM, 2.0 * p.M * static_cast<double>(p.N) * p.K);
  const auto kernel = a_unsigned ? few_rows_kernel<R, W4, true> : few_rows_kernel<R, W4, false>;
  QDIT_CUDA_CHECK(ctx, qdit_launch_overlapped(ctx, kernel, grid, dim3(ROWS_THREADS), static_cast<size_t>(R) * p.K, static_cast<const uint8_t*>(A),
                                              static_cast<const uint8_t*>(W), p));
  return qdit_after_launch(ctx, "few_rows_kernel");
}

}  // namespace

int32_t qdit_launch_few_rows(qdit_ctx* ctx, const void* A, const void* W, const qgemm::GemmParams& p, bool a_unsigned, bool packed4) {
  if (p.M == 1) return packed4 ? launch_rows<1, true>(ctx, A, W, p, a_unsigned) : launch_rows<1, false>(ctx, A, W, p, a_unsigned);
  if (p.M == 2) return packed4 ? launch_rows<2, true>(ctx, A, W, p, a_unsigned) : launch_rows<2, false>(ctx, A, W, p, a_unsigned);
  return packed4 ? launch_rows<4, true>(ctx, A, W, p, a_unsigned) : launch_rows<4, false>(ctx, A, W, p, a_unsigned);
}
