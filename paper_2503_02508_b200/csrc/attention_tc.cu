// Non-causal softmax attention on the 5th-generation tensor cores (tcgen05 kind::f16, bf16 operands), any token count
// that is a multiple of 64.
//
// What bounds it: the chain of one 128 x 128 block of scores, whose exponentials alone are 1024 clocks of the
// special-function unit (16 per clock and SM) against about 890 clocks of tensor-core work (320 for the scores; P.V runs
// at half rate because its operand A comes from tensor memory), plus four hand-overs between warps of 150-250 clocks.  So
// everything that is not the softmax itself (operand loads, both products, the output) runs in other warps, on work of the
// next or the previous block, and two chains per SM fill each other's gaps.
//
// Persistent CTA, one per SM; its work items are (sample, head, 256 queries).  The two 128-query tiles of an item are
// two independent softmax streams ("slots") that share the K and V tiles; while one slot waits for its products the
// other one has the exponentials to itself.
//   warps 0-3, 4-7   softmax of slot 0 / 1, one thread per query row: P = exp2(s * scale - m) as bf16 pairs in tensor
//                    memory, from where P.V takes its A operand
//   warps 8-11       output: accumulator -> registers, division by the row sum, 8-bit quantizer or conversion, staged
//                    per warp in shared memory and written row-contiguously
//   warp 12          TMA producer: Q double-buffered over items; a three-stage ring, each stage V of a block and K of the
//                    block after it (of the next item at an item's end)
//   warps 13, 14     tensor-core issuers of slot 0 / 1.  The scores of block j + 1 (of the next item as well) are issued as
//                    soon as the probabilities of block j are ready, before most of the product that consumes these
// Tensor memory (512 columns): per slot 128 columns of scores, 80 of accumulator and 48 for the probabilities of 96 keys;
// the probabilities of the other 32 keys go over the scores, and the product that reads them is issued before the next
// scores.  All 128 keys in columns of their own would take 544 columns; all of them over the scores would put the whole
// P.V product between a block's exponentials and the next block's.
//
// A row's exponents have its maximum so far as reference (a pass over the block's scores of its own; the accumulator is
// rescaled in tensor memory when some row of a warp has a new maximum).  8 x 16 x 1024 x 72 takes 75.1 us, 32 x 16 x 256 x 72
// 25.6; with the maximum of the first 32 keys as reference and no pass it was 58.9 and 22.2, but less exact (see `rise`).
//
// One exponential in four is a polynomial on the FMA pipe (as exact as the others, see exp2_poly): the special-function unit shares its instruction queue with
// barrier and tensor-memory operations, and with all exponentials in it a hand-over took 250-300 clocks.
//
// With no more query tiles than SMs an item is one tile, and one stream: it then has both score buffers and both places for
// probabilities to itself, so the scores of a block are ready before the exponentials of the block before it have ended, and
// the chain is the exponentials alone (ONE; the same operations in the same order, so the same bits).
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

constexpr int TQ = 128;                        // queries per slot
constexpr int TK = 128;                        // keys per block
constexpr int SM_WARPS = 8;                    // softmax warps: four per slot
constexpr int OUT_WARPS = 4;
constexpr int TC_THREADS = (SM_WARPS + OUT_WARPS + 3) * 32;
constexpr int KV_STAGES = 3;                   // a stage: V of a block and K of the block after it
constexpr int MAIN_BYTES = 128 * 128;          // 128 rows x 64 bf16, 128-byte swizzle
constexpr int TAIL_BYTES = 128 * 16;           // 128 rows x 8 bf16, no swizzle
// tensor-memory columns of slot s
__device__ __forceinline__ uint32_t col_s(int s) { return static_cast<uint32_t>(128 * s); }        // scores (128)
__device__ __forceinline__ uint32_t col_o(int s) { return static_cast<uint32_t>(256 + 64 * s); }   // accumulator, head dims 0..63
__device__ __forceinline__ uint32_t col_t(int s) { return static_cast<uint32_t>(384 + 16 * s); }   // head dims 64..71, the row sum, padding
__device__ __forceinline__ uint32_t col_p(int s) { return static_cast<uint32_t>(416 + 48 * s); }   // probabilities of 96 keys
constexpr uint32_t P_ALIAS = 112;              // score column that the probabilities of the other 32 keys start at
constexpr int STAGGER_CLOCKS = 1200;           // start of slot 1 behind slot 0

struct AttnTcParams {
  int T, H;
  int n_blk;           // key blocks of 128, the first one possibly 64 wide
  int n_qgroups;       // work items per (sample, head)
  int slots;           // query tiles per work item: 2, or 1 when there are too few tiles to fill the SMs in pairs
  int n_items;
  float scale_log2;    // softmax_scale * log2(e)
  void* out;
  int out_dtype;
  QuantArgs qa;
  int* status;
};

template <int DH>
struct TCfg {
  static constexpr bool TAIL = DH > 64;                 // head dim 72: columns 64..71 in a tile of their own
  static constexpr int OP_BYTES = MAIN_BYTES + (TAIL ? TAIL_BYTES : 0);
  // output staging per warp: 32 rows, each padded by 16 bytes (8-bit rows: 8) against bank conflicts; f32 is the widest
  static constexpr int STAGE_ROW_MAX = DH * 4 + 16;
  static constexpr int OUT_BYTES = OUT_WARPS * 32 * STAGE_ROW_MAX;
  static constexpr int TILES = 4 + 2 * KV_STAGES;       // Q: 2 buffers x 2 slots; V / K ring
  static constexpr int SMEM_BYTES = 1024 + TILES * (MAIN_BYTES + TAIL_BYTES) + 2 * TAIL_BYTES + OUT_BYTES + 512;
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

// 2^x for two values without the special-function unit: x = n + f with n the nearest integer (biased by 127 in the low
// mantissa bits of x + 1.5 * 2^23 + 127, from where it goes to the exponent field of the factor 2^n), 2^f on [-1/2, 1/2] as
// a polynomial of degree 6 with p(0) = 1 (equi-ripple fit of the relative error).  With the f32 arithmetic the error is 7.9e-8
// at most and 2.7e-8 rms, ex2.approx's measured the same way 1.4e-7 and 5.8e-8; degree 5 has 1.7e-7, degree 4 2.7e-6.  From -126.5
// down the result is zero, for -infinity too; NaN stays NaN.
__device__ __forceinline__ float2 exp2_poly(float2 x) {
  asm("max.NaN.f32 %0, %0, %1;" : "+f"(x.x) : "f"(-127.0f));
  asm("max.NaN.f32 %0, %0, %1;" : "+f"(x.y) : "f"(-127.0f));
  const float2 big = make_float2(12583039.0f, 12583039.0f), neg_big = make_float2(-12583039.0f, -12583039.0f);
  const float2 t = __fadd2_rn(x, big), n = __fadd2_rn(t, neg_big);
  const float2 f = __ffma2_rn(n, make_float2(-1.0f, -1.0f), x);
  float2 y = __ffma2_rn(make_float2(0.00015353362f, 0.00015353362f), f, make_float2(0.0013398874f, 0.0013398874f));
  y = __ffma2_rn(y, f, make_float2(0.009618437f, 0.009618437f));
  y = __ffma2_rn(y, f, make_float2(0.055503324f, 0.055503324f));
  y = __ffma2_rn(y, f, make_float2(0.24022648f, 0.24022648f));
  y = __ffma2_rn(y, f, make_float2(0.6931472f, 0.6931472f));
  y = __ffma2_rn(y, f, make_float2(1.0f, 1.0f));
  return __fmul2_rn(y, make_float2(__int_as_float(__float_as_int(t.x) << 23), __int_as_float(__float_as_int(t.y) << 23)));
}

struct Item {
  int row0, col0, q0;
};
template <int DH>
__device__ __forceinline__ Item item_of(const AttnTcParams& p, int item) {
  const int g = item % p.n_qgroups, bh = item / p.n_qgroups;
  Item it;
  it.row0 = (bh / p.H) * p.T;
  it.col0 = (bh % p.H) * DH;
  it.q0 = g * p.slots * TQ;
  return it;
}
// token of a key block's first key
__device__ __forceinline__ int key_of(const AttnTcParams& p, int j) { return j == 0 ? 0 : j * TK - (p.n_blk * TK - p.T); }
__device__ __forceinline__ bool slot_active(const AttnTcParams& p, const Item& it, int slot) {
  return slot < p.slots && it.q0 + slot * TQ < p.T;
}

template <int DH, bool ONE>
__global__ void __launch_bounds__(TC_THREADS, 1)
attention_tc_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                    const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_qt,
                    const __grid_constant__ CUtensorMap tm_kt, const __grid_constant__ CUtensorMap tm_vt,
                    const AttnTcParams p) {
  using C = TCfg<DH>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sQ = smem;                                    // [2 buffers][2 slots]
  uint8_t* sKV = sQ + 4 * MAIN_BYTES;                    // [KV_STAGES][V, K]
  uint8_t* sQt = sKV + 2 * KV_STAGES * MAIN_BYTES;       // tails, same indices
  uint8_t* sKVt = sQt + 4 * TAIL_BYTES;
  uint8_t* sZero = sKVt + 2 * KV_STAGES * TAIL_BYTES;    // constant halves of the tail steps (behind every tail tile)
  uint8_t* sOne = sZero + TAIL_BYTES;
  uint8_t* sOut = sOne + TAIL_BYTES;
  uint64_t* bars = reinterpret_cast<uint64_t*>(sOut + C::OUT_BYTES);
  uint64_t* q_full = bars;              // [2] Q tiles of an item landed (tx)
  uint64_t* q_empty = bars + 2;         // [2] all score products of the item done (commit of both issuers)
  uint64_t* kv_full = bars + 4;         // [KV_STAGES] (tx)
  uint64_t* kv_empty = kv_full + KV_STAGES;   // [KV_STAGES] (commit of both issuers)
  uint64_t* s_full = kv_empty + KV_STAGES;    // [2] scores of a slot's block complete (commit)
  // With one query tile the next two go by score buffer too, as s_full does: the softmax warps may finish two blocks before the issuer
  // has looked at the first, and one barrier would then be two phases ahead of its waiter, whose parity says "not yet" for good.
  uint64_t* p_full = s_full + 2;        // [2] probabilities written (4 warps)
  uint64_t* pv_done = p_full + 2;       // [2] P.V product complete (commit)
  uint64_t* o_full = pv_done + 2;       // [2] last P.V product of an item complete (commit)
  uint64_t* o_empty = o_full + 2;       // [2] accumulator read by the output warps (4 warps)
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(o_empty + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_holder + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int i = 0; i < 2; ++i) {
      mbar_init(&q_full[i], 1);
      mbar_init(&q_empty[i], 2);
      mbar_init(&s_full[i], 1);
      mbar_init(&p_full[i], 4);
      mbar_init(&pv_done[i], 1);
      mbar_init(&o_full[i], 1);
      mbar_init(&o_empty[i], OUT_WARPS);
    }
    for (int i = 0; i < KV_STAGES; ++i) {
      mbar_init(&kv_full[i], 1);
      mbar_init(&kv_empty[i], ONE ? 1 : 2);
    }
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
    }
  } else if (warp == SM_WARPS + OUT_WARPS + 1) {
    tmem_alloc(tmem_holder, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_holder;
  // shared and tensor memory only so far; Q, K and V come from the previous kernel of the stream
  grid_dependency_wait();
  grid_dependency_release();

  if (warp < SM_WARPS) {
    // ------------------------------------------------------------------ softmax, one thread per query row
    const int slot = warp >> 2;
    const uint32_t trow = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16);
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
    // 32 scores in registers -> P = exp2(s * scale - m) as 16 bf16 pairs; one pair in four on the FMA pipe
    auto probs = [&](const uint32_t (&v)[32], uint32_t (&pk)[16]) {
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        float2 a = __ffma2_rn(make_float2(__uint_as_float(v[2 * i]), __uint_as_float(v[2 * i + 1])), sc2, nm2);
        if ((i & 3) == 3) {
          a = exp2_poly(a);
        } else {
          a.x = ex2_approx(a.x);
          a.y = ex2_approx(a.y);
        }
        pk[i] = pack_bf16x2(a.x, a.y);
      }
    };
    uint32_t n = 0;  // blocks of this slot so far
    bool ok = true;
    for (int item = blockIdx.x; item < p.n_items && ok; item += gridDim.x) {
      if (ONE ? slot == 1 : !slot_active(p, item_of<DH>(p, item), slot)) continue;
      float m_ref = -INFINITY;
#pragma unroll 1
      for (int j = 0; j < p.n_blk; ++j, ++n) {
        const bool full = j > 0 || p.T % TK == 0;  // else 64 keys
        const bool ends = j + 1 == p.n_blk;
        const int buf = ONE ? j & 1 : slot;      // which scores and probabilities
        const uint32_t s_col = trow + col_s(buf), p_col = trow + col_p(buf);
        ok = mbar_wait_warp(&s_full[buf], (ONE ? n >> 1 : n) & 1u, abort_flag, p.status);
        if (!ok) break;
        tc_fence_after();
        auto set_reference = [&](float m) {
          m_ref = m;
          // a row of -inf: zero probabilities so far, undefined (NaN) if nothing else follows
          const float nm = m_ref == -INFINITY ? (ends ? __int_as_float(0x7FFFFFFF) : 0.0f) : -m_ref;
          nm2 = make_float2(nm, nm);
        };
        // Some row has a new maximum: move the references of the warp and rescale what has been summed.
        auto grow = [&](float mx) {
          const float m_new = fmaxf(m_ref, mx);
          const float alpha = m_new == m_ref ? 1.0f : ex2_approx(m_ref - m_new);
          set_reference(m_new);
          if (j == 0) return;
#pragma unroll 1
          for (uint32_t c = 0; c < 80; c += 16) {
            const uint32_t col = trow + (c < 64 ? col_o(slot) + c : col_t(slot));
            uint32_t v[16];
            tmem_ld_32x16(col, v);
            tmem_ld_wait();
#pragma unroll
            for (int i = 0; i < 16; ++i) v[i] = __float_as_uint(__uint_as_float(v[i]) * alpha);
            tmem_st_32x16(col, v);
          }
          tmem_st_wait();
        };
        // The previous product has read the columns that the probabilities go to, and the accumulator may be touched.  (With
        // two buffers the scores of this block were issued after the product that read its columns; the accumulator is
        // waited for where it is rescaled.)
        auto previous_done = [&](bool seen) -> bool {
          if (n == 0) return true;
          uint64_t* const done = &pv_done[ONE ? (n - 1) & 1u : slot];
          if (!__all_sync(0xffffffffu, seen) && !mbar_wait_warp(done, (ONE ? (n - 1) >> 1 : n - 1) & 1u, abort_flag, p.status)) return false;
          tc_fence_after();
          return true;
        };
        uint32_t va[32], vb[32], pa[16], pb[16];
        tmem_ld_32x32(s_col, va);
        tmem_ld_wait_for(va);
        // The largest probability of a row so far is exactly one and those near it lie below a power of two, where bf16 rounds
        // them best: a reference taken from the first 32 keys alone saves this pass, but the rounding error of N(0,1) operands
        // grows from 1.44e-3 to 1.61e-3 of the result (twice the logits: 0.86e-3 to 1.31e-3).
        auto rise = [&](float mx) -> bool {
          if (j == 0) {
            set_reference(mx);
          } else if (__any_sync(0xffffffffu, mx > m_ref)) {
            if (!previous_done(false)) return false;
            grow(mx);
          } else {
            set_reference(m_ref);
          }
          return true;
        };
        if (full) {
          tmem_ld_32x32(s_col + 32, vb);
          float mx = row_max(va, -INFINITY);
          tmem_ld_wait_for(vb);
          tmem_ld_32x32(s_col + 64, va);
          mx = row_max(vb, mx);
          tmem_ld_wait_for(va);
          tmem_ld_32x32(s_col + 96, vb);
          mx = row_max(va, mx);
          tmem_ld_wait_for(vb);
          mx = row_max(vb, mx) * p.scale_log2;
          ok = rise(mx);
          if (!ok) break;
          // the last two chunks are in registers; the first two are read again meanwhile
          probs(vb, pb);
          tmem_ld_32x32(s_col, vb);
          const bool seen = ONE || n == 0 || mbar_test_wait(&pv_done[slot], (n - 1) & 1u);
          probs(va, pa);
          tmem_ld_wait_for(vb);
          tmem_ld_32x32(s_col + 32, va);
          if (!ONE) ok = previous_done(seen);
          if (!ok) break;
          tmem_st_32x16(p_col + 32, pa);
          probs(vb, pa);
          tmem_st_32x16(p_col, pa);
          tmem_ld_wait_for(va);
          tmem_st_32x16(s_col + P_ALIAS, pb);   // all scores have been read: their columns are free
          probs(va, pb);
          tmem_st_32x16(p_col + 16, pb);
        } else {
          tmem_ld_32x32(s_col + 32, vb);
          tmem_ld_wait_for(vb);
          const float mx = row_max(vb, row_max(va, -INFINITY)) * p.scale_log2;
          ok = previous_done(false) && rise(mx);
          if (!ok) break;
          probs(va, pa);
          tmem_st_32x16(p_col, pa);
          probs(vb, pb);
          tmem_st_32x16(p_col + 16, pb);
        }
        tmem_st_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&p_full[buf]);
      }
    }
  } else if (warp < SM_WARPS + OUT_WARPS) {
    // ------------------------------------------------------------------ output
    const int quad = warp & 3;
    const uint32_t trow = tmem + (static_cast<uint32_t>(quad * 32) << 16);
    uint8_t* stage = sOut + quad * 32 * C::STAGE_ROW_MAX;
    const int64_t pitch = static_cast<int64_t>(p.H) * DH;
    float q_inv = 0.0f;
    if (p.out_dtype == QDIT_I8) q_inv = __fdiv_rn(1.0f, p.qa.scale_dev ? __ldg(p.qa.scale_dev) : p.qa.scale);
    uint32_t phases = 0u;  // bit s: parity of slot s's next tile
    bool ok = true;
    for (int item = blockIdx.x; item < p.n_items && ok; item += gridDim.x) {
      const Item it = item_of<DH>(p, item);
#pragma unroll 1
      for (int slot = 0; slot < 2; ++slot) {
        if (!slot_active(p, it, slot)) continue;
        ok = mbar_wait_warp(&o_full[slot], (phases >> slot) & 1u, abort_flag, p.status);
        if (!ok) break;
        phases ^= 1u << slot;
        tc_fence_after();
        uint32_t o[DH], w[8];
        {
          uint32_t(&lo)[32] = *reinterpret_cast<uint32_t(*)[32]>(&o[0]);
          uint32_t(&hi)[32] = *reinterpret_cast<uint32_t(*)[32]>(&o[32]);
          tmem_ld_32x32(trow + col_o(slot), lo);
          tmem_ld_32x32(trow + col_o(slot) + 32, hi);
          if constexpr (C::TAIL) {
            uint32_t(&tl)[8] = *reinterpret_cast<uint32_t(*)[8]>(&o[64]);
            tmem_ld_32x8(trow + col_t(slot), tl);
          }
          tmem_ld_32x8(trow + col_t(slot) + 8, w);
          tmem_ld_wait();
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_relaxed(&o_empty[slot]);
        const float inv_l = 1.0f / __uint_as_float(w[0]);
        const int q_first = it.q0 + slot * TQ + quad * 32;   // rows of a warp are all inside or all outside (T % 64 == 0)
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
            float y[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) y[i] = __uint_as_float(o[8 * g + i]) * inv_l;
            code[g] = quantize_pack8(y, q_inv, p.qa.zp, p.qa.qmin, p.qa.qmax);
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
    }
  } else if (warp == SM_WARPS + OUT_WARPS) {
    // ------------------------------------------------------------------ TMA producer
    int st = 0, n = 0;
    uint32_t ph = 0;
    bool ok = true;
    auto load_q = [&](const Item& it, int qb) {
      const bool two = slot_active(p, it, 1);
      if (elect_one()) {
        mbar_expect_tx(&q_full[qb], two ? 2 * C::OP_BYTES : C::OP_BYTES);
        for (int s = 0; s < (two ? 2 : 1); ++s) {
          tma_load_2d(sQ + (qb * 2 + s) * MAIN_BYTES, &tm_q, it.col0, it.row0 + it.q0 + s * TQ, &q_full[qb]);
          if (C::TAIL) tma_load_2d(sQt + (qb * 2 + s) * TAIL_BYTES, &tm_qt, it.col0 + 64, it.row0 + it.q0 + s * TQ, &q_full[qb]);
        }
      }
      __syncwarp();
    };
    // one stage: V of block jv of item vi (none for jv < 0), K of block jk of item ki (none for jk < 0)
    auto load_kv = [&](const Item& vi, int jv, const Item& ki, int jk) {
      if (!mbar_wait_warp(&kv_empty[st], ph ^ 1u, abort_flag, p.status)) { ok = false; return; }
      if (elect_one()) {
        mbar_expect_tx(&kv_full[st], (jv >= 0 && jk >= 0) ? 2 * C::OP_BYTES : C::OP_BYTES);
        if (jk >= 0) {
          tma_load_2d(sKV + (2 * st + 1) * MAIN_BYTES, &tm_k, ki.col0, ki.row0 + key_of(p, jk), &kv_full[st]);
          if (C::TAIL) tma_load_2d(sKVt + (2 * st + 1) * TAIL_BYTES, &tm_kt, ki.col0 + 64, ki.row0 + key_of(p, jk), &kv_full[st]);
        }
        if (jv >= 0) {
          tma_load_2d(sKV + 2 * st * MAIN_BYTES, &tm_v, vi.col0, vi.row0 + key_of(p, jv), &kv_full[st]);
          if (C::TAIL) tma_load_2d(sKVt + 2 * st * TAIL_BYTES, &tm_vt, vi.col0 + 64, vi.row0 + key_of(p, jv), &kv_full[st]);
        }
      }
      __syncwarp();
      if (++st == KV_STAGES) { st = 0; ph ^= 1u; }
    };
    int item = blockIdx.x;            // the grid never exceeds the number of items
    Item it = item_of<DH>(p, item);
    load_q(it, 0);
    load_kv(it, -1, it, 0);
    while (ok) {
      const int next_item = item + static_cast<int>(gridDim.x);
      const bool more = next_item < p.n_items;
      const Item nit = item_of<DH>(p, more ? next_item : item);
      for (int j = 0; j + 1 < p.n_blk && ok; ++j) load_kv(it, j, it, j + 1);
      if (more && ok) {
        const int qb = (n + 1) & 1;
        if (n >= 1 && !mbar_wait_warp(&q_empty[qb], static_cast<uint32_t>((n - 1) >> 1) & 1u, abort_flag, p.status)) { ok = false; break; }
        load_q(nit, qb);
      }
      if (ok) load_kv(it, p.n_blk - 1, nit, more ? 0 : -1);
      if (!more) break;
      item = next_item;
      it = nit;
      ++n;
    }
    if (*abort_flag) {
      // give copies already in flight time to land before the CTA's shared memory is released
      for (int i = 0; i < 2000; ++i) __nanosleep(1000);
    }
  } else {
    // ------------------------------------------------------------------ tensor-core issuers, one warp per slot (the warp
    // stays converged and one elected thread issues: with the role behind `lane == 0` an instruction took 90 clocks to
    // issue, which set the pace of the whole kernel).  Both warps walk all items and release every stage, so that a slot
    // without a query tile keeps step with the ring.
    const int slot = warp - (SM_WARPS + OUT_WARPS + 1);
    const uint32_t id_s = umma_idesc_bf16(128, TK, false), id_s_half = umma_idesc_bf16(128, TK / 2, false);
    const uint32_t id_o = umma_idesc_bf16(128, 64, true), id_ot = umma_idesc_bf16(128, 16, true);
    const uint32_t zero = smem_u32(sZero), one = smem_u32(sOne);
    const bool ragged = p.T % TK != 0;
    const uint64_t q_desc = umma_desc(smem_u32(sQ), 1024, 2), kv_desc = umma_desc(smem_u32(sKV), 1024, 2);
    const uint32_t o_acc = tmem + col_o(slot), t_acc = tmem + col_t(slot);
    // S = Q K^T: 4 k-steps of 16 out of the 64-column tiles, one out of the tails (called by the elected thread)
    auto issue_s = [&](int qb, int st, uint32_t id, int buf) {
      const uint32_t s_acc = tmem + col_s(buf);
      const uint64_t qd = q_desc + static_cast<uint64_t>((qb * 2 + slot) * (MAIN_BYTES >> 4));
      const uint64_t kd = kv_desc + static_cast<uint64_t>((2 * st + 1) * (MAIN_BYTES >> 4));
#pragma unroll
      for (int k = 0; k < 4; ++k) umma_bf16(s_acc, qd + 2 * k, kd + 2 * k, id, k ? 1u : 0u);
      if (C::TAIL) {
        const uint32_t qt = smem_u32(sQt) + static_cast<uint32_t>((qb * 2 + slot) * TAIL_BYTES);
        const uint32_t kt = smem_u32(sKVt) + static_cast<uint32_t>((2 * st + 1) * TAIL_BYTES);
        umma_bf16(s_acc, desc_plain(qt, zero - qt, 128), desc_plain(kt, zero - kt, 128), id, 1u);
      }
      umma_commit(&s_full[buf]);
    };
    // O += P V over 32 keys: two k-steps of 16; `a` = tensor-memory columns of the probabilities, g = first 16-key group.
    // Columns 64..71 of V (head dim 64: zeros) and the column of ones behind them form the 16-wide second product of a step.
    auto issue_pv = [&](int st, uint32_t a, int g, uint32_t first_acc) {
      const uint64_t vd = kv_desc + static_cast<uint64_t>(2 * st * (MAIN_BYTES >> 4));
      const uint32_t left = C::TAIL ? smem_u32(sKVt) + static_cast<uint32_t>(2 * st * TAIL_BYTES) : zero;
      const uint64_t td = desc_plain(left, 128, one - left);
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        const uint32_t acc = s == 0 ? first_acc : 1u;
        umma_bf16_ta(o_acc, a + 8 * s, vd + 128 * (g + s), id_o, acc);
        umma_bf16_ta(t_acc, a + 8 * s, td + 16 * (g + s), id_ot, acc);
      }
    };
    auto issue_pv_alias = [&](int st, int buf, uint32_t first_acc) { issue_pv(st, tmem + col_s(buf) + P_ALIAS, 6, first_acc); };
    auto issue_pv_rest = [&](int st, int buf, bool half, uint32_t first_acc) {
      const uint32_t p_op = tmem + col_p(buf);
      issue_pv(st, p_op, 0, half ? first_acc : 1u);
      issue_pv(st, p_op + 16, 2, 1u);
      if (!half) issue_pv(st, p_op + 32, 4, 1u);
    };
    if constexpr (ONE) {
      if (slot == 0) {
        // One item, one tile.  Stage t of the ring holds K of block t and V of block t - 1; scores run two blocks ahead of the
        // products.
        auto landed = [&](int t) { return mbar_wait_warp(&kv_full[t % KV_STAGES], static_cast<uint32_t>(t / KV_STAGES) & 1u, abort_flag, p.status); };
        auto scores = [&](int j) {
          if (!landed(j)) return false;
          tc_fence_after();
          if (elect_one()) {
            issue_s(0, j % KV_STAGES, (ragged && j == 0) ? id_s_half : id_s, j & 1);
            if (j == 0) umma_commit(&kv_empty[0]);
          }
          __syncwarp();
          return true;
        };
        bool ok = mbar_wait_warp(&q_full[0], 0, abort_flag, p.status) && scores(0) && (p.n_blk == 1 || scores(1));
        for (int j = 0; j < p.n_blk && ok; ++j) {
          const bool half = ragged && j == 0;
          ok = landed(j + 1) && mbar_wait_warp(&p_full[j & 1], static_cast<uint32_t>(j >> 1) & 1u, abort_flag, p.status);
          if (!ok) break;
          tc_fence_after();
          if (elect_one()) {
            const uint32_t acc0 = j == 0 ? 0u : 1u;
            const int st = (j + 1) % KV_STAGES;
            if (!half) issue_pv_alias(st, j & 1, acc0);
            issue_pv_rest(st, j & 1, half, acc0);
            umma_commit(&pv_done[j & 1]);
            if (j + 1 == p.n_blk) umma_commit(&o_full[0]);
            umma_commit(&kv_empty[st]);
          }
          __syncwarp();
          if (j + 2 < p.n_blk) ok = scores(j + 2);
        }
      }
    } else {
      int st = 0, n = 0;                    // ring position, items so far
      uint32_t ph = 0;
      uint32_t blk = 0, tiles = 0;          // blocks and query tiles of the slot so far
      auto advance = [&]() { if (++st == KV_STAGES) { st = 0; ph ^= 1u; } };
      // first scores of the first item
      int item = blockIdx.x;
      bool active = slot_active(p, item_of<DH>(p, item), slot);
      bool ok = mbar_wait_warp(&q_full[0], 0, abort_flag, p.status) && mbar_wait_warp(&kv_full[0], 0, abort_flag, p.status);
      if (ok) {
        if (slot == 1 && active) {
          // half a block behind slot 0: the slots then take turns at the tensor core and the special-function unit instead
          // of asking for both at the same time, and stay that way
          const long long t0 = clock64();
          for (int i = 0; i < 64 && clock64() - t0 < STAGGER_CLOCKS; ++i) __nanosleep(20);
        }
        tc_fence_after();
        if (elect_one()) {
          if (active) issue_s(0, st, ragged ? id_s_half : id_s, slot);
          umma_commit(&kv_empty[st]);
          if (p.n_blk == 1) umma_commit(&q_empty[0]);
        }
        __syncwarp();
        advance();
      }
      while (ok) {
        const int next_item = item + static_cast<int>(gridDim.x);
        const bool more = next_item < p.n_items;
        const bool next_active = more && slot_active(p, item_of<DH>(p, next_item), slot);
        for (int j = 0; j < p.n_blk; ++j) {
          const bool last = j + 1 == p.n_blk;
          const int jn = last ? 0 : j + 1, qn = last ? (n + 1) & 1 : n & 1;   // the score block after this one, its Q buffer
          const bool next_s = last ? next_active : active;
          // this stage (and Q of the next item) was asked for long before the probabilities are ready
          ok = mbar_wait_warp(&kv_full[st], ph, abort_flag, p.status);
          if (ok && last && more) ok = mbar_wait_warp(&q_full[qn], static_cast<uint32_t>((n + 1) >> 1) & 1u, abort_flag, p.status);
          // the accumulator is overwritten: the output warps must have read the previous tile
          if (ok && active && j == 0 && tiles > 0) ok = mbar_wait_warp(&o_empty[slot], (tiles - 1) & 1u, abort_flag, p.status);
          if (ok && active) ok = mbar_wait_warp(&p_full[slot], blk & 1u, abort_flag, p.status);
          if (!ok) break;
          tc_fence_after();
          if (elect_one()) {
            const uint32_t id = (ragged && jn == 0) ? id_s_half : id_s;
            const uint32_t acc0 = j == 0 ? 0u : 1u;
            const bool half = ragged && j == 0;
            // first the product that reads probabilities out of the score columns, then the next scores, which the softmax
            // warps wait for, then the rest
            if (active && !half) issue_pv_alias(st, slot, acc0);
            if (next_s) issue_s(qn, st, id, slot);
            if (active) {
              issue_pv_rest(st, slot, half, acc0);
              umma_commit(&pv_done[slot]);
              if (last) umma_commit(&o_full[slot]);
            }
            umma_commit(&kv_empty[st]);
            if (jn + 1 == p.n_blk && (!last || more)) umma_commit(&q_empty[qn]);
          }
          __syncwarp();
          if (active) ++blk;
          advance();
        }
        if (!more || !ok) break;
        if (active) ++tiles;
        item = next_item;
        active = next_active;
        ++n;
      }
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
  const int64_t tiles = (T + TQ - 1) / TQ, heads = static_cast<int64_t>(B) * H;
  p.slots = heads * tiles <= ctx->num_sms ? 1 : 2;   // few tiles: one per SM instead of two on half of them
  p.n_qgroups = static_cast<int>((tiles + p.slots - 1) / p.slots);
  p.n_items = static_cast<int>(heads * p.n_qgroups);
  const int grid = p.n_items < ctx->num_sms ? p.n_items : ctx->num_sms;
  ProfScope prof(ctx, QDIT_PROF_ATTENTION, 4.0 * B * H * static_cast<double>(T) * T * DH);
  const auto kernel = p.slots == 1 ? attention_tc_kernel<DH, true> : attention_tc_kernel<DH, false>;
  QDIT_TRY(qdit_allow_smem(ctx, kernel, C::SMEM_BYTES));
  QDIT_CUDA_CHECK(ctx, qdit_launch_overlapped(ctx, kernel, dim3(grid), dim3(TC_THREADS), C::SMEM_BYTES, tq, tk, tv, tqt, tkt, tvt, p));
  return qdit_after_launch(ctx, "attention_tc_kernel");
}

}  // namespace

// Tensor-core attention for T % 64 == 0 and head dim 64 or 72 (arguments already validated by qdit_attention).
int32_t qdit_launch_attention_tc(qdit_ctx* ctx, const void* q, const void* k, const void* v, int64_t ld, int B, int H,
                                 int T, int dh, float softmax_scale, void* out, int out_dtype, QuantArgs qa) {
  AttnTcParams p{};
  p.T = T;
  p.H = H;
  p.n_blk = (T + TK - 1) / TK;
  p.scale_log2 = softmax_scale * 1.4426950408889634f;
  p.out = out;
  p.out_dtype = out_dtype;
  p.qa = qa;
  p.status = ctx->d_status;
  if (dh == 64) return launch_tc<64>(ctx, q, k, v, ld, B, H, T, p);
  return launch_tc<72>(ctx, q, k, v, ld, B, H, T, p);
}
