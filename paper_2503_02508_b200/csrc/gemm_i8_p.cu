// W8A8 linear layer with many rows: a pair of CTAs (the two SMs of a cluster) computes tiles of 256 tokens x BN channels with
// tcgen05.mma.cta_group::2, token-major, BN a multiple of 32 up to 256 chosen per launch.
//
// What bounds it: one SM multiplies 8192 pairs of codes per clock and its shared memory moves 128 bytes per clock, for the operands
// that arrive and for those that the tensor core reads.  A 128 x 256 tile of one CTA takes 512 clocks of the tensor core per 128-byte
// k-block but 96 KB through shared memory (48 in, 48 out), 768 clocks.  In a pair each CTA fetches its own 128 tokens and half of the
// channels, and reads no more than those (the tensor cores exchange the halves): 64 KB, 512 clocks as well.  Measured without an
// epilogue, 8192 x 4608 x 4608: 0.30 us per k-block against 0.355 with single CTAs, 0.26 with operands that stay in shared memory.
// 8192 x 3456 x 1152 takes 24.0 us (26.9 with single CTAs), 65536 x 3456 x 1152 182-188 (222): 2.8 POP/s at 1.4 GHz, where the power cap
// leaves the clock; 8192 x 4608 x 1152 with GELU and codes 36.2 (40.1); 65536 x 1152 x 4608 gated 256 (276).
//
// CTA = 2 + EPI_WARPS warps: warp 0 TMA producer (of its own half of the operands; both CTAs' copies report to the leader's
// barrier), warp 1 MMA issuer (the leader, CTA 0 of the pair, issues for both; commits arrive in both), the others epilogue: the
// accumulator of a CTA is its 128 tokens (TMEM lanes) x BN channels (columns), two accumulator stages of 256 columns.
//
// Epilogues work on chunks of 32 tokens (a lane quadrant) x 32 channels and hand whole tiles to TMA stores:
//   16-bit and f32 outputs (classes 1, 3, 5 to 7): the accumulator is read in the matrix-fragment layout (tcgen05.ld 16x256b), in
//     which a thread holds pairs of adjacent channels of four tokens; scales, bias and gate of its eight channels are pairs of
//     registers for two-wide arithmetic, stmatrix lays the finished pairs down as swizzled rows.  The residual of the gated
//     layers comes by TMA one chunk ahead and is read with ldmatrix.
//   8-bit codes (class 2): a thread holds 32 channels of one token (tcgen05.ld 32x32b), the channels' parameters come from shared
//     memory for all lanes at once, four codes are packed into a word and the row's 32 bytes written by two stores.  A code costs
//     two operations of the special-function unit (16 per clock): 4100 clocks for 128 x 256 of them, of the 4600 that the products take
//     with K = 1152; the arithmetic alone runs in 4800 with 16 warps (6000 with 8).  So the warps share nothing but the accumulator: with a
//     barrier among them per tile the epilogue took 7600 clocks, now 6100.
// Stores by the warps themselves instead of TMA were slower in every class (QKV at 8192 rows 32 us), and so were chunks of 64 channels.
#include "gemm_common.cuh"

namespace {

using namespace qgemm;

constexpr int MAX_STAGES = 8;
constexpr int SHORT_K = 2048;                        // gated layers with a shorter reduction: class 4
constexpr int A_BYTES = 128 * BK;                    // 128 tokens of a k-block; half of the channels follow (BN / 2 rows)
constexpr int ACC_COLS = 256;

template <int EPI>
struct PCfg {
  static constexpr bool CODES = EPI == 2, GATED = EPI == 3 || EPI == 4;
  static constexpr int EPI_WARPS = CODES ? 16 : EPI == 4 ? 12 : 8;
  static constexpr int SPLIT = EPI_WARPS / 4;           // warps per lane quadrant, which take the chunks in turn
  static constexpr int THREADS = 64 + EPI_WARPS * 32;
  static constexpr int TILE_BYTES = CODES ? 1024 : 2048;                 // output tile: 32 x 32 codes or bf16, 16 x 32 f32
  // two of them, used in turn; gated: each receives the residual of a chunk and is overwritten by its output, a third one takes the
  // cache copy
  static constexpr int STAGING_PER_WARP = (GATED ? 3 : 2) * TILE_BYTES;
  static constexpr int PARAM_BYTES = CODES ? EPI_WARPS * 384 : 0;        // per warp [scale, bias, zero-point term][channel of a chunk]
  static constexpr int BAR_BYTES = 512;
  static constexpr int EXTRA_BYTES = EPI_WARPS * STAGING_PER_WARP + PARAM_BYTES + BAR_BYTES + 1024;
  static constexpr int SMEM_BYTES = 232448;              // what the other parts leave holds the stages: 5 or 6 of 256 channels, more of fewer
};

// ----------------------------------------------------------------------------- instructions of a CTA pair
__device__ __forceinline__ uint32_t pair_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void pair_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void pair_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// address of a barrier of the leader, as this CTA and its copies name it
__device__ __forceinline__ uint32_t in_leader(const void* p) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"(smem_u32(p)));
  return r;
}
__device__ __forceinline__ void arrive_at_leader(uint32_t bar) {
  asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
// Copy into this CTA's shared memory, reported to a barrier of the leader.
__device__ __forceinline__ void pair_load_2d(void* smem_dst, const void* tmap, int32_t c0, int32_t c1, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2 [%0], [%1, {%2, %3}], [%4];"
      ::"r"(smem_u32(smem_dst)), "l"(reinterpret_cast<uint64_t>(tmap)), "r"(c0), "r"(c1), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void pair_tmem_alloc(uint32_t* smem_holder, uint32_t ncols) {  // a warp of each CTA
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(smem_holder)), "r"(ncols) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void pair_tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void pair_umma_i8(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::i8 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Arrives on the barrier at this offset in both CTAs once the products issued so far have completed.
__device__ __forceinline__ void pair_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
               ::"r"(smem_u32(bar)), "h"(static_cast<uint16_t>(3))
               : "memory");
}
// Four 8 x 8 matrices of 16-bit elements, rows of 16 bytes: thread t holds, of matrix j (register j), the elements 2(t%4),
// 2(t%4) + 1 of row t/4 and supplies the address of row t%8 of matrix t/8.
__device__ __forceinline__ void stmatrix_x4(uint32_t addr, uint32_t r0, uint32_t r1, uint32_t r2, uint32_t r3) {
  asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(r0), "r"(r1), "r"(r2), "r"(r3) : "memory");
}
__device__ __forceinline__ void ldmatrix_x4(uint32_t addr, uint32_t (&r)[4]) {   // the same layout
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}

// ----------------------------------------------------------------------------- arithmetic on a pair of channels
// (the same rounded operations as in the other kernels of these layers, two at a time)
__device__ __forceinline__ float2 to_float2(uint32_t a, uint32_t b) {
  return make_float2(static_cast<float>(static_cast<int>(a)), static_cast<float>(static_cast<int>(b)));
}
// gelu_tanh_f of both (FTZ: the quotient without the handling of subnormal numbers, for codes that are zero either way)
__device__ __forceinline__ float div_approx_ftz(float a, float b) {
  float r;
  asm("div.approx.ftz.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}
template <bool FTZ>
__device__ __forceinline__ float2 gelu_tanh_f2(float2 x) {
  const float2 u = __fmul2_rn(x, __ffma2_rn(__fmul2_rn(x, x), make_float2(-0.1029432396f, -0.1029432396f), make_float2(-2.3022081998f, -2.3022081998f)));
  const float2 d = __fadd2_rn(make_float2(1.0f, 1.0f), make_float2(ex2_approx(u.x), ex2_approx(u.y)));
  if (!FTZ) return make_float2(__fdividef(x.x, d.x), __fdividef(x.y, d.y));
  return make_float2(div_approx_ftz(x.x, d.x), div_approx_ftz(x.y, d.y));
}

// Accumulators of a chunk (32 tokens x 32 channels) in fragments: a = tokens 0..15, b = tokens 16..31; the pair of channels
// 8k + 2(t%4), + 1 of token 8g + t/4.
__device__ __forceinline__ float2 frag_acc(const uint32_t (&a)[16], const uint32_t (&b)[16], int g, int k) {
  const uint32_t(&v)[16] = g < 2 ? a : b;
  return to_float2(v[4 * k + 2 * (g & 1)], v[4 * k + 2 * (g & 1) + 1]);
}

// Weights of more bytes are read once, tile by tile, and the tokens stay in L2: 1600 x 193536 x 1152 takes 399 us instead of 548, its
// 223 MB of weights being fetched once instead of seven times.
constexpr int64_t TOKENS_FIRST_BYTES = 48 << 20;

struct PairParams {
  GemmParams g;
  int bn;        // channels per tile
  int stages, stage_bytes;
  int tokens_first;
  uint32_t idesc;
};

// The epilogue of class 2 for an output step below 2^-125, at which subnormal activations have codes (see there): the codes of a warp's chunks, one
// after the other and by plain stores.  Not inlined, so that the usual loop is compiled as if this were not there.
struct TinySteps {
  uint64_t* tfull_bar;
  volatile int* abort_flag;
  uint32_t taddr, tempty0;      // this lane quadrant's rows of the accumulators; the leader's barriers that take them back
  float a_scale, o_inv;
  int pair, num_pairs, row, part, split;   // row: of this thread's token in the pair's tile
};
__device__ __noinline__ void codes_of_tiny_steps(const PairParams& pp, const TinySteps s) {
  const GemmParams& p = pp.g;
  const int chunks = pp.bn / 32, total = p.num_m_tiles * p.num_n_tiles, lane = static_cast<int>(threadIdx.x) & 31;
  int it = 0;
  for (int i = s.pair; i < total; i += s.num_pairs, ++it) {
    const int as = it & 1;
    const int m = (pp.tokens_first ? i % p.num_m_tiles : i / p.num_n_tiles) * 256 + s.row, n0 = (pp.tokens_first ? i / p.num_m_tiles : i % p.num_n_tiles) * pp.bn;
    if (!mbar_wait_warp(&s.tfull_bar[as], static_cast<uint32_t>(it >> 1) & 1u, s.abort_flag, p.status)) return;
    tc_fence_after();
    for (int c = s.part; c < chunks; c += s.split) {
      uint32_t v[32];
      __syncwarp();
      tmem_ld_32x32(s.taddr + static_cast<uint32_t>(as * ACC_COLS + c * 32), v);
      tmem_ld_wait_for(v);
#pragma unroll 1
      for (int j = 0; j < 32; ++j) {
        const int n = n0 + c * 32 + j;
        if (m >= p.M || n >= p.N) continue;
        const int acc = static_cast<int>(v[j]) - (p.a_zp != 0 ? p.a_zp * p.w_colsum[n] : 0);
        const float x = gelu_tanh_f(__fmaf_rn(static_cast<float>(acc), __fmul_rn(s.a_scale, p.w_scale[n]), p.bias[n]));
        static_cast<uint8_t*>(p.out)[static_cast<int64_t>(m) * p.ldo + n] = static_cast<uint8_t>(__float2int_rn(quantize_code(x, s.o_inv, p.o_zp, p.o_qmin, p.o_qmax)));
      }
    }
    tc_fence_before();
    __syncwarp();
    if (lane == 0) arrive_at_leader(s.tempty0 + static_cast<uint32_t>(as) * 8u);
  }
}

template <int EPI>
__global__ void __launch_bounds__(PCfg<EPI>::THREADS, 1)
gemm_i8_pair_kernel(const __grid_constant__ CUtensorMap tmap_a, const __grid_constant__ CUtensorMap tmap_w,
                    const __grid_constant__ CUtensorMap tmap_out, const __grid_constant__ CUtensorMap tmap_cache,
                    const __grid_constant__ CUtensorMap tmap_res, const __grid_constant__ PairParams pp) {
  using C = PCfg<EPI>;
  const GemmParams& p = pp.g;
  const int stages = pp.stages, stage_bytes = pp.stage_bytes;
  extern __shared__ uint8_t smem_raw[];
  // identical layout in both CTAs: the alignment slack must not depend on the CTA
  uint8_t* smem = smem_raw + (1024u - (smem_u32(smem_raw) & 1023u)) % 1024u;
  uint8_t* staging = smem + stages * stage_bytes;        // behind the stages (this CTA's tokens, its half of the channels): [EPI_WARPS][tiles]
  float* params = reinterpret_cast<float*>(staging + C::EPI_WARPS * C::STAGING_PER_WARP);
  uint64_t* full_bar = reinterpret_cast<uint64_t*>(staging + C::EPI_WARPS * C::STAGING_PER_WARP + C::PARAM_BYTES);   // leader: both halves landed (tx)
  uint64_t* empty_bar = full_bar + MAX_STAGES;               // both: stage read by the products (commit)
  uint64_t* tfull_bar = empty_bar + MAX_STAGES;              // both: accumulator complete (commit)
  uint64_t* tempty_bar = tfull_bar + 2;                  // leader: accumulator read by the epilogue warps of both CTAs
  uint64_t* res_bar = tempty_bar + 2;                    // [EPI_WARPS][2] gated: the residual of a chunk landed (tx)
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(res_bar + (C::GATED ? 2 * C::EPI_WARPS : 0));
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_holder + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = static_cast<int>(pair_rank());

  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) {
      mbar_init(&full_bar[s], 1);
      mbar_init(&empty_bar[s], 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&tfull_bar[s], 1);
      mbar_init(&tempty_bar[s], 2 * C::EPI_WARPS);
    }
    if (C::GATED) {
      for (int s = 0; s < 2 * C::EPI_WARPS; ++s) mbar_init(&res_bar[s], 1);
    }
    *abort_flag = 0;
    mbar_fence_init();
  }
  if (warp == 0) {
    if (lane == 0) {
      tma_prefetch_desc(&tmap_a);
      tma_prefetch_desc(&tmap_w);
      tma_prefetch_desc(&tmap_out);
      if (C::GATED) {
        tma_prefetch_desc(&tmap_cache);
        tma_prefetch_desc(&tmap_res);
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    pair_tmem_alloc(tmem_holder, 512);
  }
  tc_fence_before();
  __syncthreads();
  // both CTAs have started and their barriers are initialised before either signals the other's
  pair_arrive();
  pair_wait();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_holder;
  grid_dependency_wait();
  grid_dependency_release();

  const int num_kb = (p.K + BK - 1) / BK;
  const int bn = pp.bn;
  const int pair = static_cast<int>(blockIdx.x) >> 1, num_pairs = static_cast<int>(gridDim.x) >> 1;
  // Tiles run along the channels first, so that pairs running together share the tokens, or along the tokens first (tokens_first) where
  // the weights are too many to stay in L2 from one pass over them to the next.
  const bool tf = pp.tokens_first != 0;
  const int total_tiles = p.num_m_tiles * p.num_n_tiles;
  // A pair's next tile is num_pairs further on: whole lines of tiles and a rest, so that no role divides per tile.
  const int line = tf ? p.num_m_tiles : p.num_n_tiles, size = tf ? 256 : bn, across = tf ? bn : 256;
  const int step_along = (num_pairs % line) * size, step_across = (num_pairs / line) * across, span = line * size;
  struct Tile {
    int i, along, across;   // index; first channel (token) of the pair's tile, first token (channel)
  };
  auto next = [&](Tile& t) {
    t.i += num_pairs;
    t.along += step_along;
    t.across += step_across;
    if (t.along >= span) {
      t.along -= span;
      t.across += across;
    }
  };
  auto m_of = [&](const Tile& t) { return tf ? t.along : t.across; };
  auto n_of = [&](const Tile& t) { return tf ? t.across : t.along; };
  const Tile first{pair, (pair % line) * size, (pair / line) * across};
  auto wait_for = [&](bool seen, uint64_t* bar, uint32_t parity) { return seen || mbar_wait(bar, parity, abort_flag, p.status); };

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer (each CTA for itself)
    if (elect_one()) {
      const uint32_t full0 = in_leader(full_bar);
      const uint32_t tx = 2u * static_cast<uint32_t>(stage_bytes);   // both CTAs' bytes of a stage
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true, seen = true;   // seen: the stage about to be filled is known to be free
      for (Tile t = first; t.i < total_tiles && ok; next(t)) {
        const int m0 = m_of(t) + rank * 128, n0 = n_of(t) + rank * (bn / 2);
        for (int kb = 0; kb < num_kb; ++kb) {
          if (!wait_for(seen, &empty_bar[stage], phase ^ 1u)) { ok = false; break; }
          const bool wrap = stage + 1 == stages;
          seen = mbar_test_wait(&empty_bar[wrap ? 0 : stage + 1], phase ^ (wrap ? 0u : 1u));
          const uint32_t bar = full0 + static_cast<uint32_t>(stage) * 8u;
          if (rank == 0) mbar_expect_tx(&full_bar[stage], tx);
          uint8_t* const dst = smem + stage * stage_bytes;
          pair_load_2d(dst, &tmap_a, kb * BK, m0, bar);
          pair_load_2d(dst + A_BYTES, &tmap_w, kb * BK, n0, bar);
          if (++stage == stages) { stage = 0; phase ^= 1u; }
        }
      }
      if (!ok) leave_time_for_copies();
    }
    __syncwarp();
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer (the leader for both)
    if (rank == 0 && elect_one()) {
      int stage = 0;
      uint32_t phase = 0;
      int it = 0;
      bool ok = true, seen = false;   // seen: the stage about to be multiplied is known to have landed
      for (Tile t = first; t.i < total_tiles && ok; next(t), ++it) {
        const int as = it & 1;
        if (!wait_for(false, &tempty_bar[as], (static_cast<uint32_t>(it >> 1) & 1u) ^ 1u)) { ok = false; break; }
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + static_cast<uint32_t>(as * ACC_COLS);
        for (int kb = 0; kb < num_kb; ++kb) {
          if (!wait_for(seen, &full_bar[stage], phase)) { ok = false; break; }
          const bool wrap = stage + 1 == stages;
          seen = mbar_test_wait(&full_bar[wrap ? 0 : stage + 1], phase ^ (wrap ? 1u : 0u));
          tc_fence_after();
          const uint64_t a_desc = umma_desc_k_sw128(smem_u32(smem + stage * stage_bytes));
          const uint64_t b_desc = a_desc + (A_BYTES >> 4);
#pragma unroll
          for (int k = 0; k < BK / UMMA_K; ++k)
            pair_umma_i8(d_tmem, a_desc + static_cast<uint64_t>(k * (UMMA_K >> 4)), b_desc + static_cast<uint64_t>(k * (UMMA_K >> 4)),
                         pp.idesc, (kb | k) != 0 ? 1u : 0u);
          pair_commit(&empty_bar[stage]);
          if (++stage == stages) { stage = 0; phase ^= 1u; }
        }
        if (ok) pair_commit(&tfull_bar[as]);
      }
      if (!ok) leave_time_for_copies();   // (the producers may have issued their last copy before)
    }
    __syncwarp();
  } else {
    // -------------------------------------------------------------------- epilogue warps
    const int e = warp - 2, quad = warp & 3, part = e >> 2;
    const float a_scale = device_value(p.a_scale_dev, p.a_scale);
    const int chunks = bn / 32;
    const int c_last = part < chunks ? part + ((chunks - 1 - part) / C::SPLIT) * C::SPLIT : -1;   // this warp's last chunk
    uint8_t* const stg = staging + e * C::STAGING_PER_WARP;
    const uint32_t tile0 = smem_u32(stg);
    const uint32_t tempty0 = in_leader(tempty_bar);
    auto release = [&](int as) {   // this warp has read its share of the accumulator
      tc_fence_before();
      __syncwarp();
      if (elect_one()) arrive_at_leader(tempty0 + static_cast<uint32_t>(as) * 8u);
    };
    int it = 0, turn = 0;
    bool ok = true;
    if constexpr (C::CODES) {
      const float o_inv = __fdiv_rn(1.0f, device_value(p.o_scale_dev, p.o_scale));
      const float lo_f = p.o_qmin - p.o_zp, hi_f = p.o_qmax - p.o_zp;
      const uint32_t z4 = (static_cast<uint32_t>(static_cast<int>(p.o_zp)) & 0xFFu) * 0x01010101u;
      const float2 o2 = make_float2(o_inv, o_inv), magic = make_float2(12582912.0f, 12582912.0f);
      // 32-byte rows, 16-byte pieces swizzled by bit 2 of the row: the stores of eight lanes meet no bank twice
      const uint32_t row_addr = tile0 + static_cast<uint32_t>(lane) * 32u, sw = (static_cast<uint32_t>(lane) >> 2 & 1u) << 4;
      // Parameters of a chunk's channels: a lane holds those of one channel, fetched one chunk ahead, and hands them to its warp
      // through shared memory (no barrier between warps: they drift apart, and one's exponentials run beside another's loads)
      float* const sc = params + e * 96;
      float* const bi = sc + 32;
      int* const zt = reinterpret_cast<int*>(sc + 64);
      float sc_next = 0.0f, bi_next = 0.0f;
      auto fetch = [&](const Tile& t, int c) {
        const int n = n_of(t) + c * 32 + lane;
        if (t.i < total_tiles && c < chunks && n < p.N) {
          sc_next = p.w_scale[n];
          bi_next = p.bias[n];
        }
      };
      fetch(first, part);
      // A subnormal activation has a code other than zero only if a step is below 2^-125.  Such steps have a function of their own, which costs the
      // others 0.1 to 0.2 us per launch (2048 x 4608 x 1152 13.4 / 13.6, 65536 rows 280.5 / 280.6): a choice inside the loop costs 8 to 15 % (its registers
      // and its schedule are full), a second copy of it 1 %.
      if (!(o_inv <= 0x1p125f)) {   // (infinite too)
        codes_of_tiny_steps(pp, TinySteps{tfull_bar, abort_flag, tmem_base + (static_cast<uint32_t>(quad * 32) << 16), tempty0, a_scale, o_inv, pair, num_pairs,
                                          rank * 128 + quad * 32 + lane, part, C::SPLIT});
      } else
      for (Tile t = first; t.i < total_tiles && ok; next(t), ++it) {
        const int as = it & 1;
        const int row0 = m_of(t) + rank * 128 + quad * 32, n0 = n_of(t);
        if (!mbar_wait_warp(&tfull_bar[as], static_cast<uint32_t>(it >> 1) & 1u, abort_flag, p.status)) { ok = false; break; }
        tc_fence_after();
        const uint32_t taddr = tmem_base + (static_cast<uint32_t>(quad * 32) << 16) + static_cast<uint32_t>(as * ACC_COLS);
        if (c_last < 0) release(as);
#pragma unroll 1
        for (int c = part; c < chunks; c += C::SPLIT) {
          const bool live = row0 < p.M && n0 + c * 32 < p.N;   // uniform over the warp
          uint32_t v[32];
          if (live) tmem_ld_32x32(taddr + static_cast<uint32_t>(c * 32), v);
          __syncwarp();   // the last chunk's parameters have been read
          sc[lane] = __fmul_rn(a_scale, sc_next);
          bi[lane] = bi_next;
          if (p.a_zp != 0) zt[lane] = n0 + c * 32 + lane < p.N ? p.a_zp * p.w_colsum[n0 + c * 32 + lane] : 0;
          __syncwarp();
          if (c + C::SPLIT < chunks) {
            fetch(t, c + C::SPLIT);
          } else {
            Tile ahead = t;
            next(ahead);
            fetch(ahead, part);
          }
          if (live) tmem_ld_wait_for(v);
          if (c == c_last) release(as);
          if (!live) continue;
          if (p.a_zp != 0) {
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const int4 z = *reinterpret_cast<const int4*>(zt + 4 * j);
              v[4 * j] -= static_cast<uint32_t>(z.x);
              v[4 * j + 1] -= static_cast<uint32_t>(z.y);
              v[4 * j + 2] -= static_cast<uint32_t>(z.z);
              v[4 * j + 3] -= static_cast<uint32_t>(z.w);
            }
          }
          uint32_t w[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const float4 s4 = *reinterpret_cast<const float4*>(sc + 4 * j), b4 = *reinterpret_cast<const float4*>(bi + 4 * j);
            const float2 x0 = gelu_tanh_f2<true>(__ffma2_rn(to_float2(v[4 * j], v[4 * j + 1]), make_float2(s4.x, s4.y), make_float2(b4.x, b4.y)));
            const float2 x1 = gelu_tanh_f2<true>(__ffma2_rn(to_float2(v[4 * j + 2], v[4 * j + 3]), make_float2(s4.z, s4.w), make_float2(b4.z, b4.w)));
            // clip(rne(t) + z, qmin, qmax) == rne(clamp(t, qmin - z, qmax - z)) + z; adding 1.5 * 2^23 rounds to nearest-even
            // and leaves the integer in the low mantissa bits; the low byte is the stored code
            float2 t0 = __fmul2_rn(x0, o2), t1 = __fmul2_rn(x1, o2);
            t0 = __fadd2_rn(make_float2(fminf(fmaxf(t0.x, lo_f), hi_f), fminf(fmaxf(t0.y, lo_f), hi_f)), magic);
            t1 = __fadd2_rn(make_float2(fminf(fmaxf(t1.x, lo_f), hi_f), fminf(fmaxf(t1.y, lo_f), hi_f)), magic);
            w[j] = __byte_perm(__byte_perm(__float_as_uint(t0.x), __float_as_uint(t0.y), 0x0040),
                               __byte_perm(__float_as_uint(t1.x), __float_as_uint(t1.y), 0x0040), 0x5410);
            if (z4 != 0u) w[j] = __vadd4(w[j], z4);   // code + z stays inside a byte
          }
          if (elect_one()) tma_store_wait_read<1>();   // the store that used this tile two chunks ago has read it
          __syncwarp();
          const uint32_t dst = row_addr + static_cast<uint32_t>(turn) * 1024u;
          asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst + sw), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]) : "memory");
          asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst + (sw ^ 16u)), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7]) : "memory");
          fence_async_smem();
          __syncwarp();
          if (elect_one()) {
            tma_store_2d(&tmap_out, stg + turn * 1024, n0 + c * 32, row0);
            tma_store_commit();
          }
          turn ^= 1;
        }
      }
    } else {
      // row this thread addresses in stmatrix: row lane % 8 of a token group, 16-byte piece lane / 8 (64-byte swizzle)
      const uint32_t row_off = static_cast<uint32_t>(lane & 7) * 64u + ((static_cast<uint32_t>(lane >> 3) ^ (static_cast<uint32_t>(lane & 7) >> 1)) << 4);
      const int row_in_tile = rank * 128 + quad * 32;
      auto live = [&](const Tile& t, int c) { return t.i < total_tiles && c < chunks && m_of(t) + row_in_tile < p.M && n_of(t) + c * 32 < p.N; };
      auto store_tile = [&](uint32_t tile, const float2 (&x)[4][4]) {
#pragma unroll
        for (int g = 0; g < 4; ++g)
          stmatrix_x4(tile + row_off + 512u * g, pack_bf16x2(x[g][0].x, x[g][0].y), pack_bf16x2(x[g][1].x, x[g][1].y),
                      pack_bf16x2(x[g][2].x, x[g][2].y), pack_bf16x2(x[g][3].x, x[g][3].y));
      };
      // Gated: the residual of a chunk is asked for one chunk ahead, into tile `turn` or the other one
      uint64_t* const rbar = res_bar + 2 * e;
      float top = 0.0f;          // class 7: largest magnitude
      uint32_t r_phase = 0;      // of both tiles' barriers, one bit each
      bool asked = false;        // the next chunk's residual is on its way
      auto ask_residual = [&](const Tile& t, int c, int tile) {
        if (elect_one()) {
          mbar_expect_tx(&rbar[tile], 2048u);
          tma_load_2d(stg + tile * 2048, &tmap_res, n_of(t) + c * 32, m_of(t) + row_in_tile, &rbar[tile]);
        }
        asked = true;
      };
      for (Tile t = first; t.i < total_tiles && ok; next(t), ++it) {
        const int as = it & 1;
        const int row0 = m_of(t) + row_in_tile;
        if (C::GATED && !asked && live(t, part)) {
          if (elect_one()) tma_store_wait_read<0>();
          __syncwarp();
          ask_residual(t, part, turn);
        }
        const float* const gate_row = C::GATED ? p.gate + static_cast<int64_t>(row0 / p.tokens) * p.ld_gate : nullptr;   // a chunk lies inside one sample
        float rs[4];   // per-token scales of this thread's four tokens
        if constexpr (EPI == 5) {
#pragma unroll
          for (int g = 0; g < 4; ++g) {
            const int m = row0 + 8 * g + (lane >> 2);
            rs[g] = m < p.M ? p.a_scale_rows[m] : 0.0f;
          }
        }
        if (!mbar_wait_warp(&tfull_bar[as], static_cast<uint32_t>(it >> 1) & 1u, abort_flag, p.status)) { ok = false; break; }
        tc_fence_after();
        const uint32_t taddr = tmem_base + (static_cast<uint32_t>(quad * 32) << 16) + static_cast<uint32_t>(as * ACC_COLS);
        if (c_last < 0) release(as);
#pragma unroll 1
        for (int c = part; c < chunks; c += C::SPLIT) {
          const int n0 = n_of(t) + c * 32;
          const bool here = live(t, c);   // uniform over the warp
          uint32_t a[16], b[16];
          // parameters of this thread's channels n0 + 8k + 2(lane%4), + 1 (past N: those of the last pair, whose results are not stored)
          float2 sc[4], bi[4], gate[4];
          [[maybe_unused]] int2 zt[4];   // f32 output: zero-point terms
          bool landed = false;   // a look at the residual's barrier, whose phase has usually ended by now
          auto channel = [&](int k) {
            const int n = n0 + 8 * k + 2 * (lane & 3);
            return n < p.N ? n : p.N - 2;
          };
          if (here) {
            if (C::GATED) landed = mbar_test_wait(&rbar[turn], r_phase >> turn & 1u);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              sc[k] = *reinterpret_cast<const float2*>(p.w_scale + channel(k));
              bi[k] = *reinterpret_cast<const float2*>(p.bias + channel(k));
              if (C::GATED) gate[k] = *reinterpret_cast<const float2*>(gate_row + channel(k));
            }
            tmem_ld_16x256b_x4(taddr + static_cast<uint32_t>(c * 32), a);
            tmem_ld_16x256b_x4(taddr + (16u << 16) + static_cast<uint32_t>(c * 32), b);
            if (EPI >= 6 && p.a_zp != 0) {   // (while the accumulator comes; the gated layers have no registers left for it, and bf16 gains nothing)
#pragma unroll
              for (int k = 0; k < 4; ++k) zt[k] = *reinterpret_cast<const int2*>(p.w_colsum + channel(k));
            }
            tmem_ld_wait();
          }
          if (c == c_last) release(as);
          if (!here) continue;
          if (p.a_zp != 0) {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const int2 z = EPI >= 6 ? zt[k] : *reinterpret_cast<const int2*>(p.w_colsum + channel(k));
              const uint32_t z0 = static_cast<uint32_t>(p.a_zp * z.x), z1 = static_cast<uint32_t>(p.a_zp * z.y);
#pragma unroll
              for (int i = 0; i < 4; i += 2) {
                a[4 * k + i] -= z0;
                a[4 * k + i + 1] -= z1;
                b[4 * k + i] -= z0;
                b[4 * k + i + 1] -= z1;
              }
            }
          }
          float2 x[4][4];   // [token group][channel group]
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const float2 s1 = EPI == 5 ? sc[k] : __fmul2_rn(make_float2(a_scale, a_scale), sc[k]);
#pragma unroll
            for (int g = 0; g < 4; ++g)
              x[g][k] = __ffma2_rn(frag_acc(a, b, g, k), EPI == 5 ? __fmul2_rn(make_float2(rs[g], rs[g]), s1) : s1, bi[k]);
          }
          if constexpr (EPI == 7) {
            // The largest magnitude is taken of what is stored: channels past N and tokens past M hold copies and zeros
#pragma unroll
            for (int k = 0; k < 4; ++k) {
#pragma unroll
              for (int g = 0; g < 4; ++g) {
                x[g][k] = gelu_tanh_f2<false>(x[g][k]);
                if (row0 + 8 * g + (lane >> 2) < p.M && n0 + 8 * k + 2 * (lane & 3) < p.N) top = fmaxf(top, fmaxf(fabsf(x[g][k].x), fabsf(x[g][k].y)));
              }
            }
          }
          if constexpr (EPI >= 6) {
            // two tiles of 16 tokens x 32 channels of f32: 128-byte rows, 16-byte pieces swizzled by the row
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              if (elect_one()) tma_store_wait_read<1>();  // the store that used this tile one chunk ago has read it
              __syncwarp();
#pragma unroll
              for (int g = 0; g < 2; ++g) {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                  const uint32_t row = static_cast<uint32_t>(8 * g + (lane >> 2)), piece = static_cast<uint32_t>(2 * k) + (static_cast<uint32_t>(lane >> 1) & 1u);
                  asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(tile0 + h * 2048u + row * 128u + ((piece ^ (row & 7u)) << 4) + ((static_cast<uint32_t>(lane) & 1u) << 3)),
                               "f"(x[2 * h + g][k].x), "f"(x[2 * h + g][k].y)
                               : "memory");
                }
              }
              fence_async_smem();
              __syncwarp();
              if (elect_one()) {
                tma_store_2d(&tmap_out, stg + h * 2048, n0, row0 + 16 * h);
                tma_store_commit();
              }
            }
          } else if constexpr (!C::GATED) {
            if (elect_one()) tma_store_wait_read<1>();  // the store that used this tile two chunks ago has read it
            __syncwarp();
            store_tile(tile0 + turn * 2048u, x);
            fence_async_smem();
            __syncwarp();
            if (elect_one()) {
              tma_store_2d(&tmap_out, stg + turn * 2048, n0, row0);
              tma_store_commit();
            }
            turn ^= 1;
          } else {
            // the previous chunk's stores have read their tiles: the cache tile is free, and the other tile takes the next residual
            if (elect_one()) tma_store_wait_read<0>();
            __syncwarp();
            asked = false;
            if (live(t, c + C::SPLIT)) {
              ask_residual(t, c + C::SPLIT, turn ^ 1);
            } else {
              Tile ahead = t;
              next(ahead);
              if (live(ahead, part)) ask_residual(ahead, part, turn ^ 1);
            }
            if (p.flags & QDIT_EPI_CACHE_STORE) store_tile(tile0 + 2 * 2048u, x);   // the branch output before the gate
            if (!mbar_wait_seen(landed, &rbar[turn], r_phase >> turn & 1u, abort_flag, p.status)) { ok = false; break; }
            r_phase ^= 1u << turn;
            const uint32_t tile_r = tile0 + turn * 2048u;
            uint32_t r[4][4];
#pragma unroll
            for (int g = 0; g < 4; ++g) ldmatrix_x4(tile_r + row_off + 512u * g, r[g]);
            // x gate, + residual: one rounded multiply and one rounded add, as in every other kernel of this layer (the two-wide
            // forms would be contracted to one rounding)
#pragma unroll
            for (int g = 0; g < 4; ++g) {
#pragma unroll
              for (int k = 0; k < 4; ++k) {
                float r0, r1;
                unpack_bf16x2(r[g][k], r0, r1);
                x[g][k] = make_float2(__fadd_rn(__fmul_rn(x[g][k].x, gate[k].x), r0), __fadd_rn(__fmul_rn(x[g][k].y, gate[k].y), r1));
              }
            }
            __syncwarp();   // every lane has read the residual: the output takes its place
            store_tile(tile_r, x);
            fence_async_smem();
            __syncwarp();
            if (elect_one()) {
              if (p.flags & QDIT_EPI_CACHE_STORE) tma_store_2d(&tmap_cache, stg + 2 * 2048, n0, row0);
              tma_store_2d(&tmap_out, stg + turn * 2048, n0, row0);
              tma_store_commit();
            }
            turn ^= 1;
          }
        }
      }
      if (EPI == 7 && p.absmax) publish_absmax(p.absmax, top);
      if (C::GATED && !ok) leave_time_for_copies();   // residuals of this chunk and of the next one
    }
    if (elect_one()) tma_store_wait_all();
    __syncwarp();
  }

  // the neighbour may still signal this CTA's barriers, read its operands or write its accumulator until it gets here itself
  tc_fence_before();
  __syncthreads();
  pair_arrive();
  pair_wait();
  if (warp == 1) {
    tc_fence_after();
    pair_tmem_dealloc(tmem_base, 512);
  }
}

template <int EPI>
int32_t launch_p_epi(qdit_ctx* ctx, const void* A, const void* W, const GemmParams& g, bool a_unsigned, int bn) {
  using C = PCfg<EPI>;
  QDIT_TRY(qdit_allow_smem(ctx, gemm_i8_pair_kernel<EPI>, C::SMEM_BYTES));
  PairParams pp{};
  pp.g = g;
  pp.bn = bn;
  pp.stage_bytes = A_BYTES + (bn / 2) * BK;
  pp.stages = (C::SMEM_BYTES - C::EXTRA_BYTES) / pp.stage_bytes;
  if (pp.stages > MAX_STAGES) pp.stages = MAX_STAGES;
  // int32 accumulators, A = activations (signed or unsigned bytes), B = weights (signed), 256 tokens x bn channels
  pp.idesc = umma_idesc_i8(256, static_cast<uint32_t>(bn), a_unsigned);
  GemmParams& p = pp.g;
  CUtensorMap ta, tw;
  QDIT_TRY(qdit_get_tmap(ctx, A, p.M, p.K, p.K, 128, BK, 1, 1, &ta));
  QDIT_TRY(qdit_get_tmap(ctx, W, p.N, p.K, p.K, static_cast<uint32_t>(bn / 2), BK, 1, 1, &tw));
  CUtensorMap to;
  if (C::CODES) QDIT_TRY(qdit_get_tmap(ctx, p.out, p.M, p.N, p.ldo, 32, 32, 3, 1, &to));
  else if (EPI >= 6) QDIT_TRY(qdit_get_tmap(ctx, p.out, p.M, p.N, p.ldo, 16, 32, 1, 4, &to));
  else QDIT_TRY(qdit_get_tmap(ctx, p.out, p.M, p.N, p.ldo, 32, 32, 2, 2, &to));
  CUtensorMap tc = to, tr = to;
  if (C::GATED) {
    if (p.cache_out) QDIT_TRY(qdit_get_tmap(ctx, p.cache_out, p.M, p.N, p.N, 32, 32, 2, 2, &tc));
    QDIT_TRY(qdit_get_tmap(ctx, p.residual, p.M, p.N, p.ldo, 32, 32, 2, 2, &tr));
  }
  p.num_m_tiles = (p.M + 255) / 256;
  p.num_n_tiles = (p.N + bn - 1) / bn;
  pp.tokens_first = static_cast<int64_t>(p.N) * p.K > TOKENS_FIRST_BYTES && p.N > p.M;
  const int total = p.num_m_tiles * p.num_n_tiles, pairs = ctx->num_sms / 2;
  ProfScope prof(ctx, QDIT_PROF_GEMM, 2.0 * p.M * static_cast<double>(p.N) * p.K);
  QDIT_CUDA_CHECK(ctx, qdit_launch_cluster(ctx, gemm_i8_pair_kernel<EPI>, dim3(2 * (total < pairs ? total : pairs)), dim3(C::THREADS), C::SMEM_BYTES, 2,
                                           ta, tw, to, tc, tr, pp));
  return qdit_after_launch(ctx, "gemm_i8_pair_kernel");
}

// Channels per tile: the least of waves x (time of a tile) + the last tile's epilogue, in clocks.  A k-block takes 200 + 1.22 BN (512 with 256
// channels: the tensor core's own time; 434 with 192: the fill and the operand reads of shared memory), a tile 600 more; an epilogue takes `chunk` for
// 32 channels and bounds the tile where that is longer; codes no less than what four chunks take, and from five on what six and a half do (four warps
// share a lane quadrant and take a chunk each: 640 x 9728 x 512 13.4 us with 64 channels, 10.6 token-major; 2048 x 4096 x 768 15.3 / 13.0 / 12.2 / 13.7
// / 13.9 / 14.6 / 12.5 with 64 / 96 / 128 / 160 / 192 / 224 / 256); with the three warps of short gated reductions three, and five and a third for four
// or five chunks (8192 x 768 x 384 11.7 / 9.9 / 10.9 / 11.1 / 9.6 / 10.9 / 11.1).  A narrower tile has to be 4 % better: it reads the tokens more often
// (fc2 at 65536 rows: 256 us with 256 channels, 316 with 192, which this estimate puts level). Measured: 8192 x 3456 x 1152 24.4 / 24.0 / 24.0 us with
// 256 / 224 / 192 channels, 2048 rows 10.1 / 9.7 / 9.0; 8192 x 1152 x 4608 40.5 with 256, 34.8 with 192, 36.5 with 128; 1024 x 4608 x 1152 10.1 with
// 256, 9.4 with 128.
struct PairTile {
  int bn;
  double cost;
};
PairTile pick_pair_tile(const GemmParams& p, int pairs) {
  const int cls = epi_class(p.flags);
  const int chunk = cls == 1 ? 540 : cls == 2 ? 770 : cls == 3 ? (p.K < SHORT_K ? 650 : 950) : cls == 5 ? 560 : cls == 6 ? 650 : 1000;
  const int64_t mt = (p.M + 255) / 256;
  const double num_kb = (p.K + BK - 1) / BK;
  PairTile best{256, 1e30};
  const int widest = p.N > 224 ? 256 : p.N <= 64 ? 64 : (p.N + 31) / 32 * 32;
  for (int bn = widest; bn >= 64; bn -= 32) {
    const int64_t waves = (mt * ((p.N + bn - 1) / bn) + pairs - 1) / pairs;
    const int n = bn / 32;
    const double taken = cls == 2 ? (n <= 4 ? 4.0 : n < 7 ? 6.5 : n) : cls == 3 && p.K < SHORT_K ? (n <= 3 ? 3.0 : n < 6 ? 5.3 : n) : n;   // chunks, in time
    const double main = num_kb * (200.0 + 1.22 * bn), epilogue = chunk * taken;
    const double cost = static_cast<double>(waves) * ((main > epilogue ? main : epilogue) + 600.0) + epilogue;
    if (cost < best.cost * 0.96) best = PairTile{bn, cost};
  }
  return best;
}

}  // namespace

double qdit_gemm_pair_cost(const qdit_ctx* ctx, const GemmParams& p) { return pick_pair_tile(p, ctx->num_sms / 2).cost; }

int32_t qdit_launch_gemm_pair(qdit_ctx* ctx, const void* A, const void* W, const GemmParams& p, bool a_unsigned) {
  const int bn = pick_pair_tile(p, ctx->num_sms / 2).bn;
  switch (epi_class(p.flags)) {
    case 1: return launch_p_epi<1>(ctx, A, W, p, a_unsigned, bn);
    case 2: return launch_p_epi<2>(ctx, A, W, p, a_unsigned, bn);
    case 3:
      // A short reduction leaves the gated epilogue as the longer part of a tile: three warps per lane quadrant instead of two, at the
      // price of one pipeline stage (proj of XL/2 at 65536 rows: 125 -> 112 us, 5000 rows 12.0 -> 11.3)
      if (p.K < SHORT_K) return launch_p_epi<4>(ctx, A, W, p, a_unsigned, bn);
      return launch_p_epi<3>(ctx, A, W, p, a_unsigned, bn);
    case 5: return launch_p_epi<5>(ctx, A, W, p, a_unsigned, bn);
    case 7: return launch_p_epi<7>(ctx, A, W, p, a_unsigned, bn);
    default: return launch_p_epi<6>(ctx, A, W, p, a_unsigned, bn);
  }
}
