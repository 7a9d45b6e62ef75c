// Non-causal softmax attention on the 5th-generation tensor cores (tcgen05 kind::f16, bf16 operands), any token count
// that is a multiple of 64.
//
// What bounds it: the chain max -> exponentials -> hand-over -> P.V -> hand-over of a 128 x 128 block of scores.  The exponentials
// are 1024 clocks of the special-function unit (16 per clock and SM), the tensor-core work about 890 (320 for the scores; P.V runs
// at half rate because its operand A comes from tensor memory), and a look at a barrier takes 200-300 clocks while that unit is
// busy, because both use one instruction queue.  So everything that is not the softmax itself (operand loads, both products, the
// output) runs in other warps, and two groups of softmax warps take the blocks in turn.
//
// Persistent CTA, one per SM; a work item is (sample, head, 128 queries), all of one size, so that an SM has at most one item more
// than another (with items of two query tiles 8 x 16 x 1024 x 72 was 4 items of 2 on some SMs, now 7 of 1).
//   warps 0-3, 4-7   softmax of the even / odd blocks, one thread per query row: P = exp2(s * scale - m) as bf16 pairs in tensor
//                    memory, from where P.V takes its A operand.  A row's maximum so far goes from group to group through
//                    shared memory, so one group's exponentials run beside the other's
//   warps 8-11       output: accumulator -> registers, division by the row sum, 8-bit quantizer or conversion, staged
//                    per warp in shared memory and written row-contiguously
//   warp 12          TMA producer: Q double-buffered over items, rings of three K and three V tiles
//   warp 13          issuer of the scores, up to three blocks ahead (of the next item as well)
//   warp 14          issuer of the P.V products
// Tensor memory (464 of 512 columns): three buffers of 128 columns of scores, the probabilities of a block over the second half of
// its own scores (whose values are in registers by then), 80 of accumulator.  A score buffer is written again only after the
// product that reads its probabilities has completed: which of two products with different accumulators the tensor core runs
// first is not defined, so the issuer waits for it.
//
// A row's exponents have its maximum so far as reference.  The accumulator is rescaled in tensor memory when some row of a warp
// has a new maximum, at the end of the block's softmax, when the product before it has usually ended.
//
// A block takes about 1600 clocks, which is the chain through the accumulator: product complete, seen by the softmax warps (200),
// rescaled (350), seen by the issuer (250), the next product (700).  Waits in that chain poll (mbar_poll_warp), and the softmax warps
// look at their next scores before the last exponentials; the output warps, which wait long, use try_wait.  With try_wait everywhere /
// polling / and the early look: 8 x 16 x 1024 x 72 61.1 / 56.5 / 55.4 us, 32 x 16 x 256 x 72 23.2 / 20.0 / 19.8, 8 x 16 x 576 x 72 29.5 /
// 27.9 / 27.7, 1 x 16 x 1024 x 72 12.5 / 12.3 / 12.2.
//
// Tried and slower: one stream of blocks per query tile, two tiles per CTA (75 us for 8 x 16 x 1024 x 72); a quarter or half of the
// exponentials as a polynomial on the FMA pipe (+5 %, +30 %); four more warps that only rescale (2 to 5 % faster above 800 tokens,
// up to 9 % slower below 320); a fresh accumulator per block, summed in the registers of eight warps (+40 %: their
// tensor-memory reads hold up the exponentials and the issue of the products).
//
// Head dim 72 does not fill a 128-byte swizzle row: columns 0..63 are a 128-byte-swizzled tile, columns 64..71 an
// 8-column tile without swizzle, which the products read as the first half of a 16-wide step; the second half comes
// from constant tiles through the descriptor's stride: zeros for Q and K, and for V a column of ones, so the ninth column
// of the accumulator's tail is the row sum of the very bf16 probabilities that multiply V.  Head dim 64 takes the column
// of ones the same way.
//
// Token counts that leave half a tile: the first key block is 64 keys wide (not the last: the keys of an early block have a
// maximum of their own as reference, and with 64 of them the error is that of the mma.sync kernel, which moves its reference every
// 64 keys; 192 tokens of N(0,1) operands: 1.36e-3 of the result, 1.37e-3 the other way round, logits twice as large 0.83e-3
// and 0.85e-3).  The surplus query rows are computed on whatever follows and not written.
#include "common.cuh"
#include "internal.h"

namespace {

using namespace qd;

constexpr int TQ = 128;                        // queries per work item
constexpr int TK = 128;                        // keys per block
constexpr int SM_WARPS = 8;                    // softmax warps: two groups of four
constexpr int OUT_WARPS = 4;
constexpr int TC_THREADS = (SM_WARPS + OUT_WARPS + 3) * 32;
constexpr int RING = 3;                        // score buffers; K tiles and V tiles in flight
constexpr int MAIN_BYTES = 128 * 128;          // 128 rows x 64 bf16, 128-byte swizzle
constexpr int TAIL_BYTES = 128 * 16;           // 128 rows x 8 bf16, no swizzle
// tensor-memory columns
__device__ __forceinline__ uint32_t col_s(int b) { return static_cast<uint32_t>(128 * b); }        // scores of buffer b (128) ...
__device__ __forceinline__ uint32_t col_p(int b) { return static_cast<uint32_t>(128 * b + 64); }   // ... and the probabilities over their second half
constexpr uint32_t COL_O = 128 * RING;         // accumulator, head dims 0..63
constexpr uint32_t COL_T = COL_O + 64;         // head dims 64..71, the row sum, padding (16)

struct AttnTcParams {
  int T, H;
  int n_blk;           // key blocks of 128, the first one possibly 64 wide
  int n_tiles;         // query tiles per (sample, head)
  int n_items;
  float scale_log2;    // softmax_scale * log2(e)
  void* out;
  int out_dtype;
  QuantArgs qa;
  int* status;
  float* absmax;       // f32 output: takes the largest magnitude, if given
};

template <int DH>
struct TCfg {
  static constexpr bool TAIL = DH > 64;                 // head dim 72: columns 64..71 in a tile of their own
  static constexpr int OP_BYTES = MAIN_BYTES + (TAIL ? TAIL_BYTES : 0);
  // output staging per warp: 32 rows, each padded by 16 bytes (8-bit rows: 8) against bank conflicts; f32 is the widest
  static constexpr int STAGE_ROW_MAX = DH * 4 + 16;
  static constexpr int OUT_BYTES = OUT_WARPS * 32 * STAGE_ROW_MAX;
  static constexpr int TILES = 2 + 2 * RING;            // Q of two items; K and V rings
  static constexpr int SMEM_BYTES = 1024 + TILES * (MAIN_BYTES + TAIL_BYTES) + 2 * TAIL_BYTES + OUT_BYTES + 2 * TQ * 4 + 512;
};

// Shared-memory descriptor of a tile without swizzle (8-element groups of 16 bytes, 8 rows of a group contiguous):
// K-major operand: sbo = distance of 8-row groups, lbo = distance of the two 8-element halves of a k-step;
// MN-major operand: sbo = distance of 8-element groups along N, lbo = distance of 8-row groups along K.
__device__ __forceinline__ uint64_t desc_plain(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  return static_cast<uint64_t>((addr & 0x3FFFFu) >> 4) | static_cast<uint64_t>((lbo >> 4) & 0x3FFF) << 16 |
         static_cast<uint64_t>((sbo >> 4) & 0x3FFF) << 32 | static_cast<uint64_t>(1) << 46;
}

__device__ __forceinline__ float fmax3(float a, float b, float c) {
  float m;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(m) : "f"(a), "f"(b), "f"(c));
  return m;
}

struct Item {
  int row0, col0, q0;
};
template <int DH>
__device__ __forceinline__ Item item_of(const AttnTcParams& p, int item) {
  const int g = item % p.n_tiles, bh = item / p.n_tiles;
  Item it;
  it.row0 = (bh / p.H) * p.T;
  it.col0 = (bh % p.H) * DH;
  it.q0 = g * TQ;
  return it;
}
// token of a key block's first key
__device__ __forceinline__ int key_of(const AttnTcParams& p, int j) { return j == 0 ? 0 : j * TK - (p.n_blk * TK - p.T); }

template <int DH>
__global__ void __launch_bounds__(TC_THREADS, 1)
attention_tc_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                    const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_qt,
                    const __grid_constant__ CUtensorMap tm_kt, const __grid_constant__ CUtensorMap tm_vt,
                    const AttnTcParams p) {
  using C = TCfg<DH>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sQ = smem;                                    // [2]
  uint8_t* sK = sQ + 2 * MAIN_BYTES;                     // [RING]
  uint8_t* sV = sK + RING * MAIN_BYTES;                  // [RING]
  uint8_t* sQt = sV + RING * MAIN_BYTES;                 // tails, same indices
  uint8_t* sKt = sQt + 2 * TAIL_BYTES;
  uint8_t* sVt = sKt + RING * TAIL_BYTES;
  uint8_t* sZero = sVt + RING * TAIL_BYTES;              // constant halves of the tail steps (behind every tail tile)
  uint8_t* sOne = sZero + TAIL_BYTES;
  uint8_t* sOut = sOne + TAIL_BYTES;
  float* sMax = reinterpret_cast<float*>(sOut + C::OUT_BYTES);   // [2 groups][128 rows] a row's maximum up to the group's block
  uint64_t* bars = reinterpret_cast<uint64_t*>(sMax + 2 * TQ);
  uint64_t* q_empty = bars;                 // [2] all score products of the item done (commit)
  uint64_t* k_full = q_empty + 2;           // [RING] (tx); with an item's first block its Q tile
  uint64_t* k_empty = k_full + RING;        // [RING] (commit)
  uint64_t* v_full = k_empty + RING;        // [RING] (tx)
  uint64_t* v_empty = v_full + RING;        // [RING] (commit)
  uint64_t* s_full = v_empty + RING;        // [RING] scores of a block complete (commit)
  uint64_t* p_full = s_full + RING;         // [RING] probabilities written, accumulator rescaled (4 warps)
  uint64_t* pv_done = p_full + RING;        // [RING] P.V product complete (commit)
  uint64_t* max_ready = pv_done + RING;     // [2 groups][4] sMax of the group's block written by a warp
  uint64_t* o_full = max_ready + 8;         // last P.V product of an item complete (commit)
  uint64_t* o_empty = o_full + 1;           // accumulator read by the output warps (4 warps)
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(o_empty + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_holder + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // The CTA's blocks are numbered through all its items: block n of them has buffer, K and V stage n % RING, used for the
  // (n / RING)-th time, and the softmax group n % 2.
  const int items = (p.n_items - static_cast<int>(blockIdx.x) + static_cast<int>(gridDim.x) - 1) / static_cast<int>(gridDim.x);
  const int n_total = items * p.n_blk;

  if (threadIdx.x == 0) {
    for (int i = 0; i < 2; ++i) {
      mbar_init(&q_empty[i], 1);
    }
    for (int i = 0; i < RING; ++i) {
      mbar_init(&k_full[i], 1);
      mbar_init(&k_empty[i], 1);
      mbar_init(&v_full[i], 1);
      mbar_init(&v_empty[i], 1);
      mbar_init(&s_full[i], 1);
      mbar_init(&p_full[i], 4);
      mbar_init(&pv_done[i], 1);
    }
    for (int i = 0; i < 8; ++i) mbar_init(&max_ready[i], 1);
    mbar_init(o_full, 1);
    mbar_init(o_empty, OUT_WARPS);
    *abort_flag = 0;
    mbar_fence_init();
  }
  if (threadIdx.x < 128) {
    // constant tiles: a row of zeros; a row whose first element is one
    *reinterpret_cast<uint4*>(sZero + threadIdx.x * 16) = make_uint4(0u, 0u, 0u, 0u);
    *reinterpret_cast<uint4*>(sOne + threadIdx.x * 16) = make_uint4(0x3F80u, 0u, 0u, 0u);
    fence_async_smem();
  }
  if (warp == SM_WARPS + OUT_WARPS) {
    if (lane == 0) {
      tma_prefetch_desc(&tm_q);
      tma_prefetch_desc(&tm_k);
      tma_prefetch_desc(&tm_v);
      if (C::TAIL) {
        tma_prefetch_desc(&tm_qt);
        tma_prefetch_desc(&tm_kt);
        tma_prefetch_desc(&tm_vt);
      }
    }
  } else if (warp == SM_WARPS + OUT_WARPS + 1) {
    tmem_alloc(tmem_holder, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_holder;

  if (warp < SM_WARPS) {
    // ------------------------------------------------------------------ softmax, one thread per query row
    const int group = warp >> 2, quad = warp & 3;
    const uint32_t trow = tmem + (static_cast<uint32_t>(quad * 32) << 16);
    float* const own_max = sMax + group * TQ + quad * 32 + lane;
    const volatile float* const other_max = sMax + (group ^ 1) * TQ + quad * 32 + lane;
    const float2 sc2 = make_float2(p.scale_log2, p.scale_log2);
    float2 nm2 = make_float2(0.0f, 0.0f);
    auto row_max = [&](const uint32_t (&v)[32], float m) -> float {
      float m0 = fmax3(m, __uint_as_float(v[0]), __uint_as_float(v[1])), m1 = fmaxf(__uint_as_float(v[2]), __uint_as_float(v[3]));
#pragma unroll
      for (int i = 4; i < 32; i += 4) {
        m0 = fmax3(m0, __uint_as_float(v[i]), __uint_as_float(v[i + 1]));
        m1 = fmax3(m1, __uint_as_float(v[i + 2]), __uint_as_float(v[i + 3]));
      }
      return fmaxf(m0, m1);
    };
    // 32 scores in registers -> P = exp2(s * scale - m) as 16 bf16 pairs
    auto probs = [&](const uint32_t (&v)[32], uint32_t (&pk)[16]) {
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const float2 a = __ffma2_rn(make_float2(__uint_as_float(v[2 * i]), __uint_as_float(v[2 * i + 1])), sc2, nm2);
        pk[i] = pack_bf16x2(ex2_approx(a.x), ex2_approx(a.y));
      }
    };
    grid_dependency_wait();
    int j = group;   // key block of the item
    bool seen_s = false;
#pragma unroll 1
    for (int n = group; n < n_total; n += 2, j += 2) {
      while (j >= p.n_blk) j -= p.n_blk;
      const bool full = j > 0 || p.T % TK == 0;  // else 64 keys
      const int buf = n % RING;
      const uint32_t s_col = trow + col_s(buf), p_col = trow + col_p(buf);
      if (!mbar_poll_seen(seen_s, &s_full[buf], static_cast<uint32_t>(n / RING) & 1u, abort_flag, p.status)) break;
      tc_fence_after();
      uint32_t va[32], vb[32], pa[16], pb[16];
      float mx, alpha = 1.0f;
      bool grew = false, seen_pv = false;
      tmem_ld_32x32(s_col, va);
      // a look at the next barrier, whose phase usually ended half a block ago
      const bool seen_max = n == 0 || mbar_test_wait(&max_ready[(group ^ 1) * 4 + quad], static_cast<uint32_t>((n - 1) >> 1) & 1u);
      tmem_ld_wait_for(va);
      tmem_ld_32x32(s_col + 32, vb);
      mx = row_max(va, -INFINITY);
      tmem_ld_wait_for(vb);
      if (full) {
        tmem_ld_32x32(s_col + 64, va);
        mx = row_max(vb, mx);
        tmem_ld_wait_for(va);
        tmem_ld_32x32(s_col + 96, vb);
        mx = row_max(va, mx);
        tmem_ld_wait_for(vb);
      }
      mx = row_max(vb, mx) * p.scale_log2;
      // The maximum of the blocks before comes from the other group, which is half a block ahead; it is waited for at an item's
      // first block too, so that neither group can be two blocks ahead of the other's look at its barrier.
      if (!mbar_poll_seen(seen_max, &max_ready[(group ^ 1) * 4 + quad], static_cast<uint32_t>((n - 1) >> 1) & 1u, abort_flag, p.status)) break;
      if (j > 0) {
        const float before = *other_max;
        grew = __any_sync(0xffffffffu, mx > before);
        mx = fmaxf(before, mx);
        alpha = mx == before ? 1.0f : ex2_approx(before - mx);
      }
      *own_max = mx;
      __syncwarp();
      if (lane == 0) mbar_arrive(&max_ready[group * 4 + quad]);
      {
        // a row of -inf: zero probabilities so far, undefined (NaN) if nothing else follows
        const float nm = mx == -INFINITY ? (j + 1 == p.n_blk ? __int_as_float(0x7FFFFFFF) : 0.0f) : -mx;
        nm2 = make_float2(nm, nm);
      }
      if (full) {
        // the last two chunks are in registers and their columns free; the first two are read again meanwhile
        probs(vb, pb);
        tmem_ld_32x32(s_col, vb);
        tmem_st_32x16(p_col + 48, pb);
        probs(va, pa);
        tmem_ld_wait_for(vb);
        tmem_ld_32x32(s_col + 32, va);
        tmem_st_32x16(p_col + 32, pa);
        probs(vb, pb);
        tmem_st_32x16(p_col, pb);
        tmem_ld_wait_for(va);
        // looks at the barriers behind this block: the scores of the group's next one and the previous product
        seen_s = n + 2 < n_total && mbar_test_wait(&s_full[(n + 2) % RING], static_cast<uint32_t>((n + 2) / RING) & 1u);
        seen_pv = grew && mbar_test_wait(&pv_done[(n - 1) % RING], static_cast<uint32_t>((n - 1) / RING) & 1u);
        probs(va, pa);
        tmem_st_32x16(p_col + 16, pa);
      } else {
        seen_s = false;
        probs(va, pa);
        tmem_st_32x16(p_col, pa);
        probs(vb, pb);
        tmem_st_32x16(p_col + 16, pb);
      }
      if (grew) {
        // some row of the warp has a new maximum: rescale what has been summed, once the previous product has added its part
        if (!mbar_poll_seen(seen_pv, &pv_done[(n - 1) % RING], static_cast<uint32_t>((n - 1) / RING) & 1u, abort_flag, p.status)) break;
        tc_fence_after();
        tmem_ld_32x32(trow + COL_O, va);
        tmem_ld_32x32(trow + COL_O + 32, vb);
        tmem_ld_32x16(trow + COL_T, pa);
        tmem_ld_wait_for(va);
#pragma unroll
        for (int i = 0; i < 32; ++i) va[i] = __float_as_uint(__uint_as_float(va[i]) * alpha);
        tmem_ld_wait_for(vb);
#pragma unroll
        for (int i = 0; i < 32; ++i) vb[i] = __float_as_uint(__uint_as_float(vb[i]) * alpha);
#pragma unroll
        for (int i = 0; i < 16; ++i) pa[i] = __float_as_uint(__uint_as_float(pa[i]) * alpha);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          tmem_st_32x16(trow + COL_O + 16 * h, *reinterpret_cast<uint32_t(*)[16]>(&va[16 * h]));
          tmem_st_32x16(trow + COL_O + 32 + 16 * h, *reinterpret_cast<uint32_t(*)[16]>(&vb[16 * h]));
        }
        tmem_st_32x16(trow + COL_T, pa);
      }
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&p_full[buf]);
    }
  } else if (warp < SM_WARPS + OUT_WARPS) {
    // ------------------------------------------------------------------ output
    const int quad = warp & 3;
    const uint32_t trow = tmem + (static_cast<uint32_t>(quad * 32) << 16);
    uint8_t* stage = sOut + quad * 32 * C::STAGE_ROW_MAX;
    const int64_t pitch = static_cast<int64_t>(p.H) * DH;
    float q_inv = 0.0f;
    grid_dependency_wait();
    grid_dependency_release();
    if (p.out_dtype == QDIT_I8) q_inv = __fdiv_rn(1.0f, device_value(p.qa.scale_dev, p.qa.scale));
#pragma unroll 1
    for (int i = 0; i < items; ++i) {
      const Item it = item_of<DH>(p, static_cast<int>(blockIdx.x) + i * static_cast<int>(gridDim.x));
      if (!mbar_wait_warp(o_full, static_cast<uint32_t>(i) & 1u, abort_flag, p.status)) break;
      tc_fence_after();
      uint32_t o[DH], w[8];
      {
        uint32_t(&lo)[32] = *reinterpret_cast<uint32_t(*)[32]>(&o[0]);
        uint32_t(&hi)[32] = *reinterpret_cast<uint32_t(*)[32]>(&o[32]);
        tmem_ld_32x32(trow + COL_O, lo);
        tmem_ld_32x32(trow + COL_O + 32, hi);
        if constexpr (C::TAIL) {
          uint32_t(&tl)[8] = *reinterpret_cast<uint32_t(*)[8]>(&o[64]);
          tmem_ld_32x8(trow + COL_T, tl);
        }
        tmem_ld_32x8(trow + COL_T + 8, w);
        tmem_ld_wait();
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_relaxed(o_empty);
      const float inv_l = 1.0f / __uint_as_float(w[0]);
      const int q_first = it.q0 + quad * 32;   // rows of a warp are all inside or all outside (T % 64 == 0)
      if (q_first >= p.T) continue;
      const int64_t base = (static_cast<int64_t>(it.row0) + q_first) * pitch + it.col0;
      if (p.out_dtype == QDIT_I8) {
        // Rows of DH bytes.  Everything that goes through the memory-instruction queue waits behind the exponentials there
        // (this piece of work took 2600 clocks with 8-byte pieces, and the other slot's accumulator was read that much later),
        // so the rows move in 16-byte pieces: head dim 72 with an even number of heads is four of them and one of 8 bytes,
        // which comes first in odd heads, whose columns start at 8 modulo 16.
        constexpr int ROW = 80;
        uint2 code[DH / 8];
#pragma unroll
        for (int g = 0; g < DH / 8; ++g) {
          float t[8];
#pragma unroll
          for (int i = 0; i < 8; i += 2) {   // two-wide products, each rounded as in quantize_pack8
            const float2 y = __fmul2_rn(make_float2(__uint_as_float(o[8 * g + i]), __uint_as_float(o[8 * g + i + 1])), make_float2(inv_l, inv_l));
            const float2 s = __fmul2_rn(y, make_float2(q_inv, q_inv));
            t[i] = s.x;
            t[i + 1] = s.y;
          }
          code[g] = quantize_pack8_scaled(t, p.qa.zp, p.qa.qmin, p.qa.qmax);
        }
        uint8_t* gout = static_cast<uint8_t*>(p.out) + base;
        const uint32_t shift = static_cast<uint32_t>(it.col0) & 8u;   // DH = 72 and an odd head
        if (DH % 16 == 0 || (p.H & 1) == 0) {
          uint8_t* srow = stage + lane * ROW;
          if (DH % 16 == 0 || shift == 0) {
#pragma unroll
            for (int g = 0; g + 1 < DH / 8; g += 2) *reinterpret_cast<uint4*>(srow + 8 * g) = make_uint4(code[g].x, code[g].y, code[g + 1].x, code[g + 1].y);
            if (DH % 16 != 0) *reinterpret_cast<uint2*>(srow + DH - 8) = code[DH / 8 - 1];
          } else {
            *reinterpret_cast<uint2*>(srow + 8) = code[0];
#pragma unroll
            for (int g = 1; g + 1 < DH / 8; g += 2) *reinterpret_cast<uint4*>(srow + 8 + 8 * g) = make_uint4(code[g].x, code[g].y, code[g + 1].x, code[g + 1].y);
          }
          __syncwarp();
          constexpr int WIDE = DH / 16;   // 16-byte pieces of a row
#pragma unroll
          for (int k = 0; k < WIDE; ++k) {
            const int r = (k * 32 + lane) / WIDE, c = (k * 32 + lane) % WIDE * 16 + static_cast<int>(shift);
            *reinterpret_cast<uint4*>(gout + r * pitch + c) = *reinterpret_cast<const uint4*>(stage + r * ROW + c + shift);
          }
          if (DH % 16 != 0) {
            const int c = shift ? 0 : DH - 8;
            *reinterpret_cast<uint2*>(gout + lane * pitch + c) = *reinterpret_cast<const uint2*>(srow + c + shift);
          }
        } else {
#pragma unroll
          for (int g = 0; g < DH / 8; ++g) *reinterpret_cast<uint2*>(gout + lane * pitch + 8 * g) = code[g];
        }
      } else if (p.out_dtype == QDIT_BF16) {
        constexpr int ROW = DH * 2 + 16, PIECES = DH / 8;
#pragma unroll
        for (int g = 0; g < DH / 8; ++g) {
          float y[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) y[i] = __uint_as_float(o[8 * g + i]) * inv_l;
          *reinterpret_cast<uint4*>(stage + lane * ROW + 16 * g) = pack_bf16x8(y);
        }
        __syncwarp();
        __nv_bfloat16* gout = static_cast<__nv_bfloat16*>(p.out) + base;
#pragma unroll 3
        for (int k = 0; k < PIECES; ++k) {
          const int i = k * 32 + lane, r = i / PIECES, c = i % PIECES;
          *reinterpret_cast<uint4*>(gout + r * pitch + 8 * c) = *reinterpret_cast<const uint4*>(stage + r * ROW + 16 * c);
        }
      } else {
        constexpr int ROW = DH * 4 + 16, PIECES = DH / 4;
        if (p.absmax) {   // (rounding is monotonic: the largest product is that of the largest magnitude)
          float m = 0.0f;
#pragma unroll
          for (int i = 0; i < DH; ++i) m = fmaxf(m, fabsf(__uint_as_float(o[i])));
          publish_absmax(p.absmax, fmaxf(m * inv_l, 0.0f));
        }
#pragma unroll
        for (int g = 0; g < DH / 4; ++g)
          *reinterpret_cast<float4*>(stage + lane * ROW + 16 * g) =
              make_float4(__uint_as_float(o[4 * g]) * inv_l, __uint_as_float(o[4 * g + 1]) * inv_l,
                          __uint_as_float(o[4 * g + 2]) * inv_l, __uint_as_float(o[4 * g + 3]) * inv_l);
        __syncwarp();
        float* gout = static_cast<float*>(p.out) + base;
#pragma unroll 3
        for (int k = 0; k < PIECES; ++k) {
          const int i = k * 32 + lane, r = i / PIECES, c = i % PIECES;
          *reinterpret_cast<float4*>(gout + r * pitch + 4 * c) = *reinterpret_cast<const float4*>(stage + r * ROW + 16 * c);
        }
      }
      __syncwarp();  // the staging rows are rewritten for the next tile
    }
  } else if (warp == SM_WARPS + OUT_WARPS) {
    // ------------------------------------------------------------------ TMA producer: K runs two blocks ahead of V
    Item k_item = item_of<DH>(p, static_cast<int>(blockIdx.x)), v_item = k_item;
    int ki = 0, kj = 0, vi = 0, vj = 0;   // item and key block of the next K and V tile
    bool ok = true;
    asm volatile("" : "+r"(k_item.row0), "+r"(k_item.col0), "+r"(k_item.q0));   // the divisions of item_of stay in front of the wait
    // Q, K and V come from the previous kernel of the stream; everything before this is done while that one still runs (with the wait
    // in front of the roles the first copy left 1200-1500 clocks after it, which one image at 256 tokens waits for)
    grid_dependency_wait();
    for (int t = 0; t < n_total + 2 && ok; ++t) {
      if (t < n_total) {
        const int st = t % RING, qb = ki & 1;
        if (kj == 0 && ki >= 2) ok = mbar_poll_warp(&q_empty[qb], static_cast<uint32_t>((ki - 2) >> 1) & 1u, abort_flag, p.status);
        if (ok && t >= RING) ok = mbar_poll_warp(&k_empty[st], static_cast<uint32_t>(t / RING - 1) & 1u, abort_flag, p.status);
        if (!ok) break;
        if (elect_one()) {
          mbar_expect_tx(&k_full[st], kj == 0 ? 2 * C::OP_BYTES : C::OP_BYTES);
          if (kj == 0) {
            tma_load_2d(sQ + qb * MAIN_BYTES, &tm_q, k_item.col0, k_item.row0 + k_item.q0, &k_full[st]);
            if (C::TAIL) tma_load_2d(sQt + qb * TAIL_BYTES, &tm_qt, k_item.col0 + 64, k_item.row0 + k_item.q0, &k_full[st]);
          }
          tma_load_2d(sK + st * MAIN_BYTES, &tm_k, k_item.col0, k_item.row0 + key_of(p, kj), &k_full[st]);
          if (C::TAIL) tma_load_2d(sKt + st * TAIL_BYTES, &tm_kt, k_item.col0 + 64, k_item.row0 + key_of(p, kj), &k_full[st]);
        }
        __syncwarp();
        if (++kj == p.n_blk) {
          kj = 0;
          ++ki;
          k_item = item_of<DH>(p, static_cast<int>(blockIdx.x) + ki * static_cast<int>(gridDim.x));
        }
      }
      if (t >= 2) {
        const int n = t - 2, st = n % RING;
        if (n >= RING) ok = mbar_poll_warp(&v_empty[st], static_cast<uint32_t>(n / RING - 1) & 1u, abort_flag, p.status);
        if (!ok) break;
        if (elect_one()) {
          mbar_expect_tx(&v_full[st], C::OP_BYTES);
          tma_load_2d(sV + st * MAIN_BYTES, &tm_v, v_item.col0, v_item.row0 + key_of(p, vj), &v_full[st]);
          if (C::TAIL) tma_load_2d(sVt + st * TAIL_BYTES, &tm_vt, v_item.col0 + 64, v_item.row0 + key_of(p, vj), &v_full[st]);
        }
        __syncwarp();
        if (++vj == p.n_blk) {
          vj = 0;
          ++vi;
          v_item = item_of<DH>(p, static_cast<int>(blockIdx.x) + vi * static_cast<int>(gridDim.x));
        }
      }
    }
    if (*abort_flag) {
      // give copies already in flight time to land before the CTA's shared memory is released
      for (int i = 0; i < 2000; ++i) __nanosleep(1000);
    }
  } else if (warp == SM_WARPS + OUT_WARPS + 1) {
    // ------------------------------------------------------------------ issuer of the scores S = Q K^T (both issuing warps stay
    // converged and one elected thread issues: with the role behind `lane == 0` an instruction took 90 clocks to issue)
    const uint32_t id_s = umma_idesc_bf16(128, TK, false), id_s_half = umma_idesc_bf16(128, TK / 2, false);
    const uint32_t zero = smem_u32(sZero);
    const bool ragged = p.T % TK != 0;
    const uint64_t q_desc = umma_desc(smem_u32(sQ), 1024, 2), k_desc = umma_desc(smem_u32(sK), 1024, 2);
    int i = 0, j = 0;   // item and key block of block n
    grid_dependency_wait();
    for (int n = 0; n < n_total; ++n) {
      const int b = n % RING, qb = i & 1;
      const uint32_t use = static_cast<uint32_t>(n / RING) & 1u;
      if (!mbar_poll_warp(&k_full[b], use, abort_flag, p.status)) break;
      // The buffer held the probabilities of block n - RING: that product has to be complete (the order in which the tensor core
      // executes two products with different accumulators is not defined).
      if (n >= RING && !mbar_poll_warp(&pv_done[b], use ^ 1u, abort_flag, p.status)) break;
      tc_fence_after();
      const bool last = j + 1 == p.n_blk;
      if (elect_one()) {
        // 4 k-steps of 16 out of the 64-column tiles, one out of the tails
        const uint32_t id = (ragged && j == 0) ? id_s_half : id_s, s_acc = tmem + col_s(b);
        const uint64_t qd = q_desc + static_cast<uint64_t>(qb * (MAIN_BYTES >> 4)), kd = k_desc + static_cast<uint64_t>(b * (MAIN_BYTES >> 4));
#pragma unroll
        for (int k = 0; k < 4; ++k) umma_bf16(s_acc, qd + 2 * k, kd + 2 * k, id, k ? 1u : 0u);
        if (C::TAIL) {
          const uint32_t qt = smem_u32(sQt) + static_cast<uint32_t>(qb * TAIL_BYTES), kt = smem_u32(sKt) + static_cast<uint32_t>(b * TAIL_BYTES);
          umma_bf16(s_acc, desc_plain(qt, zero - qt, 128), desc_plain(kt, zero - kt, 128), id, 1u);
        }
        umma_commit(&s_full[b]);
        umma_commit(&k_empty[b]);
        if (last) umma_commit(&q_empty[qb]);
      }
      __syncwarp();
      if (last) { j = 0; ++i; } else { ++j; }
    }
  } else {
    // ------------------------------------------------------------------ issuer of the products O += P V
    const uint32_t id_o = umma_idesc_bf16(128, 64, true), id_ot = umma_idesc_bf16(128, 16, true);
    const uint32_t zero = smem_u32(sZero), one = smem_u32(sOne);
    const bool ragged = p.T % TK != 0;
    const uint64_t v_desc = umma_desc(smem_u32(sV), 1024, 2);
    const uint32_t o_acc = tmem + COL_O, t_acc = tmem + COL_T;
    int i = 0, j = 0;
    grid_dependency_wait();
    for (int n = 0; n < n_total; ++n) {
      const int b = n % RING;
      const uint32_t use = static_cast<uint32_t>(n / RING) & 1u;
      if (!mbar_poll_warp(&v_full[b], use, abort_flag, p.status)) break;
      // the accumulator is overwritten: the output warps must have read the previous item's
      if (j == 0 && i > 0 && !mbar_poll_warp(o_empty, static_cast<uint32_t>(i - 1) & 1u, abort_flag, p.status)) break;
      if (!mbar_poll_warp(&p_full[b], use, abort_flag, p.status)) break;
      tc_fence_after();
      const bool last = j + 1 == p.n_blk, half = ragged && j == 0;
      if (elect_one()) {
        // k-steps of 16 keys; columns 64..71 of V (head dim 64: zeros) and the column of ones behind them form the 16-wide
        // second product of a step
        const uint32_t a = tmem + col_p(b);
        const uint64_t vd = v_desc + static_cast<uint64_t>(b * (MAIN_BYTES >> 4));
        const uint32_t left = C::TAIL ? smem_u32(sVt) + static_cast<uint32_t>(b * TAIL_BYTES) : zero;
        const uint64_t td = desc_plain(left, 128, one - left);
        auto step = [&](int g, uint32_t acc) {
          umma_bf16_ta(o_acc, a + 8 * g, vd + 128 * g, id_o, acc);
          umma_bf16_ta(t_acc, a + 8 * g, td + 16 * g, id_ot, acc);
        };
        step(0, j == 0 ? 0u : 1u);
#pragma unroll
        for (int g = 1; g < 4; ++g) step(g, 1u);
        if (!half) {
#pragma unroll
          for (int g = 4; g < 8; ++g) step(g, 1u);
        }
        umma_commit(&pv_done[b]);
        umma_commit(&v_empty[b]);
        if (last) umma_commit(o_full);
      }
      __syncwarp();
      if (last) { j = 0; ++i; } else { ++j; }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == SM_WARPS + OUT_WARPS + 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

template <int DH>
int32_t launch_tc(qdit_ctx* ctx, const void* q, const void* k, const void* v, int64_t ld, int B, int H, int T, AttnTcParams& p) {
  using C = TCfg<DH>;
  const uint64_t rows = static_cast<uint64_t>(B) * T, cols = static_cast<uint64_t>(H) * DH;
  CUtensorMap tq, tk, tv, tqt, tkt, tvt;
  QDIT_TRY(qdit_get_tmap(ctx, q, rows, cols, ld, 128, 64, 1, 2, &tq));
  QDIT_TRY(qdit_get_tmap(ctx, k, rows, cols, ld, 128, 64, 1, 2, &tk));
  QDIT_TRY(qdit_get_tmap(ctx, v, rows, cols, ld, 128, 64, 1, 2, &tv));
  tqt = tq;
  tkt = tk;
  tvt = tv;
  if (C::TAIL) {
    QDIT_TRY(qdit_get_tmap(ctx, q, rows, cols, ld, 128, 8, 0, 2, &tqt));
    QDIT_TRY(qdit_get_tmap(ctx, k, rows, cols, ld, 128, 8, 0, 2, &tkt));
    QDIT_TRY(qdit_get_tmap(ctx, v, rows, cols, ld, 128, 8, 0, 2, &tvt));
  }
  p.n_tiles = (T + TQ - 1) / TQ;
  p.n_items = static_cast<int>(static_cast<int64_t>(B) * H * p.n_tiles);
  const int grid = p.n_items < ctx->num_sms ? p.n_items : ctx->num_sms;
  ProfScope prof(ctx, QDIT_PROF_ATTENTION, 4.0 * B * H * static_cast<double>(T) * T * DH);
  QDIT_TRY(qdit_allow_smem(ctx, attention_tc_kernel<DH>, C::SMEM_BYTES));
  QDIT_CUDA_CHECK(ctx, qdit_launch_overlapped(ctx, attention_tc_kernel<DH>, dim3(grid), dim3(TC_THREADS), C::SMEM_BYTES, tq, tk, tv, tqt, tkt, tvt, p));
  return qdit_after_launch(ctx, "attention_tc_kernel");
}

}  // namespace

// Tensor-core attention for T % 64 == 0 and head dim 64 or 72 (arguments already validated by qdit_attention).
int32_t qdit_launch_attention_tc(qdit_ctx* ctx, const void* q, const void* k, const void* v, int64_t ld, int B, int H,
                                 int T, int dh, float softmax_scale, void* out, int out_dtype, QuantArgs qa, float* absmax) {
  AttnTcParams p{};
  p.T = T;
  p.H = H;
  p.n_blk = (T + TK - 1) / TK;
  p.scale_log2 = softmax_scale * 1.4426950408889634f;
  p.out = out;
  p.out_dtype = out_dtype;
  p.qa = qa;
  p.status = ctx->d_status;
  p.absmax = absmax;
  if (dh == 64) return launch_tc<64>(ctx, q, k, v, ld, B, H, T, p);
  return launch_tc<72>(ctx, q, k, v, ld, B, H, T, p);
}
