// W8A8 linear layer: persistent tcgen05 kind::i8 GEMM with TMEM int32 accumulators and a fused
// de-quantising epilogue (bias / GELU / cache store / adaLN gate / residual / re-quantisation).
//
// CTA = 2 + NUM_EPI_WARPS warps: warp 0  TMA producer  (A and W tiles -> 128B-swizzled smem ring, mbarrier tx)
//                 warp 1  MMA issuer    (tcgen05.mma into one of two TMEM accumulator stages)
//                 warps 2..      epilogue      (EPI_SPLIT warps per TMEM lane quadrant, taking 32-column chunks in turn)
// The two accumulator stages let the epilogue of tile i overlap the main loop of tile i+1.
// Tiles are 128 x BN, K is consumed in blocks of 128 bytes (4 MMAs of K = 32 each).
//
// Epilogue data flow per 32x32 chunk: tcgen05.ld gives each thread one ROW of the chunk, which is the
// wrong shape for global memory (32 lanes -> 32 different lines).  The raw accumulators are therefore
// transposed through a 4 KB XOR-swizzled shared-memory patch per warp; afterwards lane (r, g) owns 8
// consecutive columns g of rows r, r+8, r+16, r+24, so that every global load/store instruction of the
// warp covers 8 rows x 64..128 contiguous bytes, and the per-column parameters (scales, bias, gate) sit
// in registers for the whole chunk.
#include "gemm_common.cuh"

namespace {

using namespace qgemm;

template <int BN>
struct Cfg {
  static constexpr int A_BYTES = BM * BK;
  static constexpr int B_BYTES = BN * BK;
  static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
  static constexpr int BAR_BYTES = 256;
  static constexpr int SMEM_LIMIT = 232448;  // 227 KB per CTA
  static constexpr int STAGES_FIT = (SMEM_LIMIT - 1024 - BAR_BYTES - STAGING_BYTES) / STAGE_BYTES;
  static constexpr int STAGES = STAGES_FIT > 8 ? 8 : STAGES_FIT;
  static constexpr int TMEM_COLS = 2 * BN <= 128 ? 128 : (2 * BN <= 256 ? 256 : 512);
  static constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + STAGING_BYTES + BAR_BYTES + 1024;  // + alignment slack
};

// PREFETCH: see epilogue_tile
template <int BN, int EPI, bool PREFETCH>
__global__ void __launch_bounds__(NUM_THREADS, 1)
gemm_i8_kernel(const __grid_constant__ CUtensorMap tmap_a, const __grid_constant__ CUtensorMap tmap_w,
               const GemmParams p, const uint32_t idesc) {
  using C = Cfg<BN>;
  constexpr int STAGES = C::STAGES;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sA = smem;
  uint8_t* sB = smem + STAGES * C::A_BYTES;
  uint8_t* staging = smem + STAGES * C::STAGE_BYTES;
  uint64_t* full_bar = reinterpret_cast<uint64_t*>(staging + STAGING_BYTES);
  uint64_t* empty_bar = full_bar + STAGES;
  uint64_t* tfull_bar = empty_bar + STAGES;
  uint64_t* tempty_bar = tfull_bar + 2;
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(tempty_bar + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_holder + 1);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full_bar[s], 1);
      mbar_init(&empty_bar[s], 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&tfull_bar[s], 1);
      mbar_init(&tempty_bar[s], NUM_EPI_WARPS);
    }
    *abort_flag = 0;
    mbar_fence_init();
  }
  if (warp == 0) {
    if (lane == 0) {
      tma_prefetch_desc(&tmap_a);
      tma_prefetch_desc(&tmap_w);
    }
  } else if (warp == 1) {
    tmem_alloc(tmem_holder, C::TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_holder;
  // Everything above touched only this CTA's shared and tensor memory.  The roles that read what the previous kernel of the stream wrote
  // wait for it themselves.

  const int num_kb = (p.K + BK - 1) / BK;
  const int total_tiles = p.num_m_tiles * p.num_n_tiles;

  // One elected thread runs each of the two roles, so that the operands of its instructions stay in uniform registers.  (Behind
  // `lane == 0` 8192 x 1152 x 4608 takes 40.1 us, with the whole warp in the role and an election at each issue 41.5, so 38.0;
  // 700 x 1152 x 4608 13.3, 11.5 and 8.2.)  With the small tiles of few rows the roles look at their next barrier before they issue
  // the current stage (9.6 us without that); 192 columns per stage leave the time, and the look costs 1 %.
  constexpr bool AHEAD = BN != 192;
  auto wait_for = [&](bool seen, uint64_t* bar, uint32_t parity) { return seen || mbar_wait(bar, parity, abort_flag, p.status); };
  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    if (elect_one()) {
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true, seen = true;   // seen: the stage about to be filled is known to be free
      // the first stages' weights come while the previous kernel still runs
      int ahead = 0;
      if (p.early && static_cast<int>(blockIdx.x) < total_tiles) {
        const int n0 = (static_cast<int>(blockIdx.x) % p.num_n_tiles) * BN;
        for (; ahead < STAGES && ahead < num_kb; ++ahead) {
          mbar_expect_tx(&full_bar[ahead], C::STAGE_BYTES);
          tma_load_2d(sB + ahead * C::B_BYTES, &tmap_w, ahead * BK, n0, &full_bar[ahead]);
        }
      }
      grid_dependency_wait();
      if (ahead > 0) {
        const int m0 = (static_cast<int>(blockIdx.x) / p.num_n_tiles) * BM;
        for (; stage < ahead; ++stage) tma_load_2d(sA + stage * C::A_BYTES, &tmap_a, stage * BK, m0, &full_bar[stage]);
        if (stage == STAGES) { stage = 0; phase ^= 1u; seen = false; }
      }
      int kb = ahead;
      for (int tile = blockIdx.x; tile < total_tiles && ok; tile += gridDim.x, kb = 0) {
        const int m0 = (tile / p.num_n_tiles) * BM;
        const int n0 = (tile % p.num_n_tiles) * BN;
        for (; kb < num_kb; ++kb) {
          if (!wait_for(seen, &empty_bar[stage], phase ^ 1u)) { ok = false; break; }
          const bool wrap = stage + 1 == STAGES;
          seen = AHEAD && mbar_test_wait(&empty_bar[wrap ? 0 : stage + 1], phase ^ (wrap ? 0u : 1u));
          mbar_expect_tx(&full_bar[stage], C::STAGE_BYTES);
          tma_load_2d(sA + stage * C::A_BYTES, &tmap_a, kb * BK, m0, &full_bar[stage]);
          tma_load_2d(sB + stage * C::B_BYTES, &tmap_w, kb * BK, n0, &full_bar[stage]);
          if (++stage == STAGES) { stage = 0; phase ^= 1u; }
        }
      }
      if (!ok) {
        // give copies already in flight time to land before the CTA's shared memory is released
        for (int i = 0; i < 2000; ++i) __nanosleep(1000);
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    if (elect_one()) {
      int stage = 0;
      uint32_t phase = 0;
      int it = 0;
      bool ok = true, seen = false;   // seen: the stage about to be multiplied is known to have landed
      for (int tile = blockIdx.x; tile < total_tiles && ok; tile += gridDim.x, ++it) {
        const int as = it & 1;
        const uint32_t aphase = static_cast<uint32_t>(it >> 1) & 1u;
        if (!wait_for(false, &tempty_bar[as], aphase ^ 1u)) { ok = false; break; }
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + static_cast<uint32_t>(as * BN);
        for (int kb = 0; kb < num_kb; ++kb) {
          if (!wait_for(seen, &full_bar[stage], phase)) { ok = false; break; }
          const bool wrap = stage + 1 == STAGES;
          seen = AHEAD && mbar_test_wait(&full_bar[wrap ? 0 : stage + 1], phase ^ (wrap ? 1u : 0u));
          tc_fence_after();
          const uint64_t a_desc = umma_desc_k_sw128(smem_u32(sA + stage * C::A_BYTES));
          const uint64_t b_desc = umma_desc_k_sw128(smem_u32(sB + stage * C::B_BYTES));
#pragma unroll
          for (int k = 0; k < BK / UMMA_K; ++k) {
            // advancing K by 32 bytes inside the swizzle row = +2 in the (address >> 4) field
            umma_i8(d_tmem, a_desc + static_cast<uint64_t>(k * (UMMA_K >> 4)),
                    b_desc + static_cast<uint64_t>(k * (UMMA_K >> 4)), idesc, (kb | k) != 0 ? 1u : 0u);
          }
          umma_commit(&empty_bar[stage]);  // frees the smem stage once these MMAs have read it
          if (++stage == STAGES) { stage = 0; phase ^= 1u; }
        }
        if (ok) umma_commit(&tfull_bar[as]);  // accumulator complete
      }
    }
  } else {
    // -------------------------------------------------------------------- epilogue warps
    const int e = warp - 2;
    const int quad = warp & 3;   // TMEM lane quadrant this warp may access
    const int half = e >> 2;     // this warp takes chunks half, half + EPI_SPLIT, ...
    const uint32_t stg = smem_u32(staging + e * (32 * 128));  // [32 rows][8 x 16 B], 16-byte index XOR (row & 7)
    if (!PREFETCH || !p.early_params) grid_dependency_wait();
    if (!PREFETCH) grid_dependency_release();
    const float a_scale = device_value(p.a_scale_dev, p.a_scale);
    float o_inv = 0.0f;
    if (epi_flags<EPI>(p) & QDIT_EPI_QUANT_OUT) o_inv = __fdiv_rn(1.0f, device_value(p.o_scale_dev, p.o_scale));
    float top = 0.0f;
    int it = 0;
    for (int tile = blockIdx.x; tile < total_tiles; tile += gridDim.x, ++it) {
      const int as = it & 1;
      const uint32_t aphase = static_cast<uint32_t>(it >> 1) & 1u;
      const int m0 = (tile / p.num_n_tiles) * BM;
      const int n0 = (tile % p.num_n_tiles) * BN;
      ChunkInputs cur;   // of this warp's chunk
      if (PREFETCH) {
        const int n = n0 + half * 32 + (lane & 3) * 8, row_base = m0 + quad * 32;
        if (half < BN / 32) prefetch_params<EPI>(p, n, row_base, a_scale, cur);
        if (it == 0) {
          if (p.early_params) grid_dependency_wait();
          grid_dependency_release();
        }
        if (half < BN / 32) prefetch_residual<EPI>(p, n, row_base, lane >> 2, cur);
      }
      if (!mbar_wait(&tfull_bar[as], aphase, abort_flag, p.status)) break;
      __syncwarp();
      tc_fence_after();
      uint64_t* release_bar = &tempty_bar[as];
      epilogue_tile<BN, EPI, PREFETCH>(p, tmem_base + static_cast<uint32_t>(as * BN), m0, n0, quad, half, stg, lane, a_scale, o_inv, cur, top,
                        [release_bar]() { mbar_arrive_relaxed(release_bar); });
    }
    __syncwarp();
    if (EPI == 7) publish_absmax(p.absmax, top);
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, C::TMEM_COLS);
  }
}

template <int BN, int EPI, bool PREFETCH>
int32_t launch_tiles(qdit_ctx* ctx, const void* A, const void* W, GemmParams& p, bool a_unsigned) {
  using C = Cfg<BN>;
  QDIT_TRY(qdit_allow_smem(ctx, gemm_i8_kernel<BN, EPI, PREFETCH>, C::SMEM_BYTES));
  CUtensorMap ta, tw;
  QDIT_TRY(qdit_get_tmap(ctx, A, p.M, p.K, p.K, BM, BK, 1, 1, &ta));
  QDIT_TRY(qdit_get_tmap(ctx, W, p.N, p.K, p.K, BN, BK, 1, 1, &tw));
  const int total = p.num_m_tiles * p.num_n_tiles;
  const int grid = total < ctx->num_sms ? total : ctx->num_sms;
  const uint32_t idesc = umma_idesc_i8(BM, BN, a_unsigned);
  ProfScope prof(ctx, QDIT_PROF_GEMM, 2.0 * p.M * static_cast<double>(p.N) * p.K);
  QDIT_CUDA_CHECK(ctx, qdit_launch_overlapped(ctx, gemm_i8_kernel<BN, EPI, PREFETCH>, dim3(grid), dim3(NUM_THREADS), C::SMEM_BYTES, ta, tw, p, idesc));
  return qdit_after_launch(ctx, "gemm_i8_kernel");
}

template <int BN, int EPI>
int32_t launch_gemm_epi(qdit_ctx* ctx, const void* A, const void* W, GemmParams& p, bool a_unsigned) {
  p.num_m_tiles = (p.M + BM - 1) / BM;
  p.num_n_tiles = (p.N + BN - 1) / BN;
  if (EPI == 1 || EPI == 2 || p.num_m_tiles * p.num_n_tiles <= ctx->num_sms) return launch_tiles<BN, EPI, true>(ctx, A, W, p, a_unsigned);
  return launch_tiles<BN, EPI, false>(ctx, A, W, p, a_unsigned);
}

template <int BN>
int32_t launch_gemm(qdit_ctx* ctx, const void* A, const void* W, GemmParams& p, bool a_unsigned) {
  switch (epi_token_major(p, ctx->opt[QDIT_OPT_GEMM_GENERIC_EPILOGUE] != 0)) {
    case 1: return launch_gemm_epi<BN, 1>(ctx, A, W, p, a_unsigned);
    case 2: return launch_gemm_epi<BN, 2>(ctx, A, W, p, a_unsigned);
    case 3: return launch_gemm_epi<BN, 3>(ctx, A, W, p, a_unsigned);
    case 7: return launch_gemm_epi<BN, 7>(ctx, A, W, p, a_unsigned);
    default: return launch_gemm_epi<BN, 0>(ctx, A, W, p, a_unsigned);
  }
}

// Tile width: prefer 192 (divides every DiT-XL/2 layer width); fall back to narrower tiles when that
// fills the SMs better.  Cost model: waves * (BN + fixed per-tile overhead).
int pick_bn(int M, int N, int num_sms, int forced) {
  if (forced == 64 || forced == 128 || forced == 192) return forced;
  const int mt = (M + BM - 1) / BM;
  int best = 192;
  double best_cost = 1e30;
  const int cands[3] = {192, 128, 64};
  for (int bn : cands) {
    const int tiles = mt * ((N + bn - 1) / bn);
    const int waves = (tiles + num_sms - 1) / num_sms;
    const double cost = static_cast<double>(waves) * (bn + 24);
    if (cost < best_cost * 0.85) {  // measured: the wider tile wins unless the narrower one saves a whole wave or more
      best_cost = cost;
      best = bn;
    }
  }
  return best;
}

// CTAs that share the reduction of a 128 x 64 tile: the most for which all clusters are resident at once (a second wave
// would cost more than the split gains: 256 x 1152 x 4608 takes 13.7 us with 36 clusters of 4, 7.4 with 36 of 3), if each CTA keeps two
// k-blocks and is spared `spare` of them.  A k-block costs the whole-reduction kernel 0.11 us and the exchange about two: 20.
// (Whole / split: 256 x 1152 x 4608 7.9 / 7.4 us with 24 spared, 512 x 1152 x 4608 8.1 / 8.5 with 18, 512 x 1152 x 2304 5.5 / 6.3,
// 256 x 1152 x 1152 5.0 / 5.6.)  Two cases gain more: with packed weights the whole-reduction kernel widens them at 0.3 us per
// k-block, and the epilogues with run-time flags (f32 output, per-token scales) are slow on one SM, whereas a cluster splits the
// epilogue too (f32 output, 256 x 384 x 1536: 6.4 / 5.3 us, 256 x 1152 x 1152: 6.1 / 5.8): 6.
constexpr int SPLIT_SPARE = 20, SPLIT_SPARE_SLOW = 6;
int pick_split(qdit_ctx* ctx, int M, int N, int K, int spare) {
  const int64_t tiles = static_cast<int64_t>((M + BM - 1) / BM) * ((N + 63) / 64);
  const int num_kb = (K + BK - 1) / BK;
  for (int s : {6, 4, 3, 2})
    if (num_kb >= 2 * s && num_kb - (num_kb + s - 1) / s >= spare && tiles * s <= ctx->num_sms && tiles <= qdit_gemm_sk_clusters(ctx, s)) return s;
  return 1;
}

constexpr int FEW_ROWS_K = 4608;   // (four rows, tensor core / streamed: 24 x 8192 6.5 / 7.9 us, 24 x 4608 5.5 / 5.0)

}  // namespace

// Both linear layers: `packed4` = W holds 4-bit codes two per byte ([N, K/2]); `w8_scratch` = optional [N, K] int8
// matrix the packed weights of a many-row layer are widened into first; `early`, `early_params`, `absmax`: see GemmParams.
int32_t qdit_linear_impl(qdit_ctx* ctx, const void* A, const void* W, int64_t M, int64_t N, int64_t K, qdit_qparams a_qp,
                         const float* a_scale_dev, uint32_t flags, const qdit_epilogue* epi, void* out, int64_t ldo,
                         bool packed4, void* w8_scratch, bool early, bool early_params, float* absmax) {
  if (!ctx) return QDIT_ERR_INVALID_ARG;
  if (M < 0 || N < 0 || K < 0) return qdit_fail(ctx, QDIT_ERR_SHAPE, "negative size");
  if (M == 0 || N == 0) return QDIT_OK;
  if (!A || !W || !out) return qdit_fail(ctx, QDIT_ERR_INVALID_ARG, "A, W or out is NULL");
  if (K == 0 || K % 16 != 0 || K > 32768) return qdit_fail(ctx, QDIT_ERR_SHAPE, "K = %lld must be a positive multiple of 16, at most 32768", static_cast<long long>(K));
  if (packed4 && K % 32 != 0) return qdit_fail(ctx, QDIT_ERR_SHAPE, "K = %lld must be a multiple of 32 for packed 4-bit weights", static_cast<long long>(K));
  if (packed4 && (flags & QDIT_EPI_ROW_SCALE)) return qdit_fail(ctx, QDIT_ERR_UNSUPPORTED, "per-token scales are not available with packed 4-bit weights");
  if (w8_scratch && !aligned16(w8_scratch)) return qdit_fail(ctx, QDIT_ERR_ALIGN, "the weight scratch must be 16-byte aligned");
  if (N % 8 != 0) return qdit_fail(ctx, QDIT_ERR_SHAPE, "N = %lld must be a multiple of 8", static_cast<long long>(N));
  if (M > (1 << 30) || N > (1 << 30)) return qdit_fail(ctx, QDIT_ERR_SHAPE, "M or N too large");
  const uint32_t out_modes = flags & (QDIT_EPI_OUT_BF16 | QDIT_EPI_OUT_F32 | QDIT_EPI_OUT_I32 | QDIT_EPI_QUANT_OUT);
  if (out_modes == 0 || (out_modes & (out_modes - 1)) != 0)
    return qdit_fail(ctx, QDIT_ERR_INVALID_ARG, "exactly one of OUT_BF16, OUT_F32, OUT_I32, QUANT_OUT must be set");
  if ((flags & QDIT_EPI_OUT_I32) && (flags & ~QDIT_EPI_OUT_I32))
    return qdit_fail(ctx, QDIT_ERR_INVALID_ARG, "OUT_I32 returns raw accumulators and takes no other flag");
  if (ldo < N) return qdit_fail(ctx, QDIT_ERR_SHAPE, "ldo smaller than N");
  if (!aligned16(A) || !aligned16(W) || !aligned16(out)) return qdit_fail(ctx, QDIT_ERR_ALIGN, "A, W and out must be 16-byte aligned");
  const int64_t osz = (flags & QDIT_EPI_QUANT_OUT) ? 1 : (flags & QDIT_EPI_OUT_BF16) ? 2 : 4;
  if ((ldo * osz) % 8 != 0 || ((flags & QDIT_EPI_QUANT_OUT) == 0 && (ldo * osz) % 16 != 0))
    return qdit_fail(ctx, QDIT_ERR_ALIGN, "row pitch of out must be a multiple of 16 bytes (8 for byte output)");
  QDIT_TRY(qdit_check_qparams(ctx, &a_qp, a_scale_dev != nullptr));
  const bool a_unsigned = a_qp.qmin >= 0 && a_qp.qmax > 127;

  GemmParams p{};
  p.M = static_cast<int>(M);
  p.N = static_cast<int>(N);
  p.K = static_cast<int>(K);
  p.flags = flags;
  p.a_scale = a_qp.scale;
  p.a_scale_dev = a_scale_dev;
  p.a_zp = a_qp.zero_point;
  p.out = out;
  p.ldo = ldo;
  p.status = ctx->d_status;
  p.tokens = 1;
  p.early = early;
  p.early_params = early_params;
  p.absmax = absmax;
  if (absmax && epi_class(flags) != 7) return qdit_fail(ctx, QDIT_ERR_INVALID_ARG, "the largest magnitude is found behind bias and GELU with f32 output only");
  if (!(flags & QDIT_EPI_OUT_I32)) {
    if (!epi || !epi->w_scale) return qdit_fail(ctx, QDIT_ERR_INVALID_ARG, "epilogue with w_scale is required");
    if (!aligned16(epi->w_scale)) return qdit_fail(ctx, QDIT_ERR_ALIGN, "w_scale must be 16-byte aligned");
    p.w_scale = epi->w_scale;
    if (a_qp.zero_point != 0) {
      if (!epi->w_colsum) return qdit_fail(ctx, QDIT_ERR_INVALID_ARG, "w_colsum is required with a non-zero activation zero point");
      if (!aligned16(epi->w_colsum)) return qdit_fail(ctx, QDIT_ERR_ALIGN, "w_colsum must be 16-byte aligned");
      p.w_colsum = epi->w_colsum;
    }
    if (flags & QDIT_EPI_BIAS) {
      if (!epi->bias) return qdit_fail(ctx, QDIT_ERR_INVALID_ARG, "BIAS set but bias is NULL");
      if (!aligned16(epi->bias)) return qdit_fail(ctx, QDIT_ERR_ALIGN, "bias must be 16-byte aligned");
      p.bias = epi->bias;
    }
    if (flags & QDIT_EPI_GATE) {
      if (!epi->gate || epi->tokens_per_sample <= 0) return qdit_fail(ctx, QDIT_ERR_INVALID_ARG, "GATE needs gate and tokens_per_sample > 0");
      if (!aligned16(epi->gate) || epi->ld_gate % 4 != 0) return qdit_fail(ctx, QDIT_ERR_ALIGN, "gate must be 16-byte aligned with ld_gate a multiple of 4");
      p.gate = epi->gate;
      p.ld_gate = epi->ld_gate;
      p.tokens = static_cast<int>(epi->tokens_per_sample);
    }
    if (flags & QDIT_EPI_RESIDUAL) {
      if (!epi->residual) return qdit_fail(ctx, QDIT_ERR_INVALID_ARG, "RESIDUAL set but residual is NULL");
      if (!aligned16(epi->residual) || ldo % 8 != 0) return qdit_fail(ctx, QDIT_ERR_ALIGN, "residual must be 16-byte aligned (base and row pitch ldo)");
      p.residual = static_cast<const __nv_bfloat16*>(epi->residual);
    }
    if (flags & QDIT_EPI_CACHE_STORE) {
      if (!epi->cache_out) return qdit_fail(ctx, QDIT_ERR_INVALID_ARG, "CACHE_STORE set but cache_out is NULL");
      if (!aligned16(epi->cache_out)) return qdit_fail(ctx, QDIT_ERR_ALIGN, "cache_out must be 16-byte aligned");
      p.cache_out = static_cast<__nv_bfloat16*>(epi->cache_out);
    }
    if (flags & QDIT_EPI_ROW_SCALE) {
      if (!epi->a_scale_rows) return qdit_fail(ctx, QDIT_ERR_INVALID_ARG, "ROW_SCALE set but a_scale_rows is NULL");
      if (a_qp.zero_point != 0) return qdit_fail(ctx, QDIT_ERR_INVALID_ARG, "ROW_SCALE needs a symmetric activation quantizer (zero_point 0)");
      p.a_scale_rows = epi->a_scale_rows;
      p.a_scale = 1.0f;
      p.a_scale_dev = nullptr;
    }
    if (flags & QDIT_EPI_QUANT_OUT) {
      QDIT_TRY(qdit_check_qparams(ctx, &epi->out_qp, epi->out_scale_dev != nullptr));
      p.o_scale = epi->out_qp.scale;
      p.o_scale_dev = epi->out_scale_dev;
      p.o_zp = static_cast<float>(epi->out_qp.zero_point);
      p.o_qmin = static_cast<float>(epi->out_qp.qmin);
      p.o_qmax = static_cast<float>(epi->out_qp.qmax);
    }
  }
  // One to four rows, f32 output (the modulation of as many images): the weights are streamed past the rows instead of through the tensor core (us, 1
  // and 4 rows, tensor core / streamed: 193536 x 1152 51.2 / 35.1 and 51.4 / 45.4, packed 4-bit weights 73.0 / 22.1 and 75.9 / 47.7; 6912 x 1152 7.0 /
  // 2.8 and 7.0 / 4.2; 1152 x 4608 7.1 / 4.1 and 7.2 / 5.7; 1152 x 384 3.4 / 2.2 and 3.3 / 2.6).  Beyond four the dot products take longer than the
  // weights; with three and four rows they do so for many channels of a short reduction too (tensor core / streamed: 193536 x 128 17.6 / 28.1, 65536 x
  // 384 10.7 / 12.2, 24576 x 256 5.1 / 5.7; packed 193536 x 64 25.2 / 30.7, 65536 x 384 12.9 / 14.5; but 65536 x 768 13.5 / 13.7 and x 1024 17.0 /
  // 15.1, 30720 x 384 7.8 / 6.6, 30720 x 32 7.3 / 6.1, packed 65536 x 512 14.4 / 12.9, 65536 x 32 12.3 / 11.2).
  const bool many_short = p.M > 2 && (p.N >= 49152 ? (packed4 ? p.K >= 64 && p.K < 512 : p.K < 768) : p.N > 16384 && !packed4 && p.K >= 96 && p.K < 384);
  if (epi_class(p.flags) == 6 && p.M <= FEW_ROWS && !p.absmax && !many_short && p.K <= FEW_ROWS_K && ctx->opt[QDIT_OPT_GEMM_BN] == 0 && ctx->opt[QDIT_OPT_GEMM_T] == 0 &&
      !ctx->opt[QDIT_OPT_GEMM_GENERIC_EPILOGUE])
    return qdit_launch_few_rows(ctx, A, W, p, a_unsigned, packed4);
  if (packed4) {
    // many rows: the layer is bound by the tensor core and its epilogue, so the weights are widened once into the
    // scratch matrix and the W8A8 kernels run on it; few rows (or no scratch): the weight bytes bound the layer and
    // the kernel that widens them in front of the tensor core reads half of them
    if (w8_scratch && M >= 1024) {
      QDIT_TRY(qdit_unpack_weight_int4(ctx, W, N, K, w8_scratch));
      W = w8_scratch;
      p.early = false;
    } else {
      // (few tiles split by the same rule as below: 256 / 512 x 1152 x 4608 take 8.5 / 10.3 us against 17.7 / 17.9)
      const int split = ctx->opt[QDIT_OPT_GEMM_BN] == 0 ? pick_split(ctx, p.M, p.N, p.K, SPLIT_SPARE_SLOW) : 1;
      return split > 1 ? qdit_launch_gemm_sk(ctx, A, W, p, a_unsigned, split, true) : qdit_launch_gemm_w4(ctx, A, W, p, a_unsigned);
    }
  }
  // QDIT_OPT_GEMM_T forces the channel-major kernel with 128 x bt tiles (its un-specialised epilogue knows no per-token
  // scales)
  const int cls = epi_class(p.flags);
  const bool row_scale = (flags & QDIT_EPI_ROW_SCALE) != 0;
  if (!row_scale && ctx->opt[QDIT_OPT_GEMM_T] != 0) return qdit_launch_gemm_t(ctx, A, W, p, a_unsigned, ctx->opt[QDIT_OPT_GEMM_T]);
  // Kernel choice.  A layer whose 128 x 192 tiles fill no more than one wave runs token-major, one CTA per tile (below): pairs gain
  // nothing there, with short reductions or long ones (us, single CTAs / pairs: 2048 x 3456 x 384 4.8 / 5.0, 1024 x 1152 x 1152 gated 5.3 / 6.5, 2048 x
  // 1152 x 4608 gated 11.7 / 11.8, 3072 rows 13.7 / 14.8).  From the second wave on pairs of CTAs are faster (QKV of XL/2 2048 rows 11.0 / 9.0, 8192
  // 26.7 / 24.0, 65536 222 / 182; fc1 40.1 / 35.4 and 310 / 270; fc2 5000 rows 31.2 / 24.4, 65536 276 / 252; proj 14.9 / 11.3 and 117 / 105).  Per-token
  // scales and f32 output take pairs earlier, because their token-major epilogue decides at run time what to do (512 x 3456 x 1152: 8.6 / 5.9 and 8.2 /
  // 6.4), unless the split reduction, which splits the epilogue too, serves them.  Layers of few columns, or of rows just right for it, fill the chip better
  // with the 128 x 256 channel-major tiles of single CTAs, at 620 clocks per k-block, 600 per tile and 4500 for the last epilogue (channel-major / pairs: QKV
  // 1280 rows 7.2 / 7.7 us, with per-token scales 11.0 / 12.1; gated 4096 rows proj 9.1 / 10.0, fc2 17.4 / 18.3; level at 8192 rows, without / with a cache
  // copy: proj 13.3 / 13.2 and 15.5 / 14.8, fc2 33.8 / 34.0 and 37.8 / 37.6, with 4-bit codes 34.2 / 35.9; 16384 rows fc2 66.0 / 67.8 and 73.0 / 75.0).
  if (ctx->opt[QDIT_OPT_GEMM_BN] == 0 && !ctx->opt[QDIT_OPT_GEMM_GENERIC_EPILOGUE]) {
    // (8-bit rows leave through TMA stores of whole 16-byte pieces, and a 32-token chunk of a gated layer has one gate row)
    const bool staged = cls == 1 || cls == 5 || cls == 6 || cls == 7 || (cls == 2 && p.N % 16 == 0 && ldo % 16 == 0) || (cls == 3 && p.tokens % 32 == 0);
    const bool slow = cls >= 5;
    const bool one_wave = static_cast<int64_t>((p.M + BM - 1) / BM) * ((p.N + 191) / 192) <= ctx->num_sms;
    if (staged && p.M >= 1024 && (cls == 3 ? p.N >= 1024 && !one_wave : (cls == 1 || cls == 5 || cls == 6) && p.N >= 2304)) {
      const int64_t waves = (static_cast<int64_t>((p.M + 255) / 256) * ((p.N + 127) / 128) + ctx->num_sms - 1) / ctx->num_sms;
      // (the epilogue of a gated tile, which also reads the residual, takes at least 4750 clocks, and bounds the tile where the reduction is short: channel-
      // major / pairs, 5000 x 4608 x 16 33.0 / 27.7 us, 4096 x 3464 x 512 30.9 / 26.0, 5000 x 3456 x 1024 25.8 / 22.0; but 16384 x 1152 x 512 20.5 / 27.0, 8192 x
      // 4608 x 384 41.6 / 43.5)
      const double products = (p.K + BK - 1) / BK * 620.0 + 600.0, tile = cls == 3 && products < 4750.0 ? 4750.0 : products;
      const double cost = static_cast<double>(waves) * tile + 4500.0;
      // (a pair's start beyond that of a single CTA; with one wave nothing hides it.  Channel-major / pairs, bf16: 1024 x 4608 x 2048 9.1 / 10.5 us,
      // 2048 x 2304 x 3072 11.4 / 12.8, 1301 x 3456 x 512 6.5 / 7.4, but 1536 x 6912 x 768 13.8 / 12.0; gated: 4096 x 1152 x 1152 9.8 / 10.9.  Nor does
      // a pair's k-block take less than a single CTA's then: 1426 x 3072 x 4608 15.0 / 16.2, per-token scales 1024 x 4096 x 3072 12.2 / 13.0, 1024 x
      // 4608 x 4096 14.5 / 15.6)
      // (a zero point costs a gated pair's epilogue up to 10 %, whose registers hold nothing ahead; a channel-major thread has one channel: 8192 x 3456
      // x 1152 39.8 / 44.5, 2048 x 4096 x 1024 13.0 / 14.1, but 4096 x 4608 x 1488 40.5 / 32.8, 6144 x 1152 x 3072 21.9 / 18.2)
      const double pairs = qdit_gemm_pair_cost(ctx, p) * (cls == 3 && p.a_zp != 0 ? 1.05 : 1.0);
      const double spare = cls == 3 ? (waves == 1 ? 3000.0 : 0.0) : cls != 1 || one_wave ? 1500.0 : waves == 1 ? 3000.0 : 2500.0;
      const double first = waves == 1 ? (p.K + BK - 1) / BK * 110.0 : 0.0;
      // (f32 output: with one wave, with two or three that are almost full, and with reductions short enough that the output's own time counts: a
      // tile's 128 channels are whole 512-byte pieces of a row there, which memory takes at 5.4 TB/s, where a pair's 128-byte pieces reach 3.4; us,
      // channel-major / pairs: 10000 x 20480 x 64 151 / 242, 6144 x 20480 x 384 98 / 152, 8192 x 6912 x 384 44 / 53, 4096 x 30720 x 768 127 / 169, 4611
      // x 15448 x 1024 83 / 94, 8192 x 9216 x 1024 88 / 95, 2048 x 30720 x 1152 78 / 86, 1728 x 4608 x 256 8.8 / 9.8, 2048 x 4096 x 768 11.0 / 12.0,
      // 3072 x 4096 x 768 14.7 / 16.2; but 3072 x 3456 x 768 14.1 / 12.2, 5000 x 4608 x 768 29.8 / 26, 8192 x 3456 x 1152 38.5 / 34.8, and 1600 x 98304
      // x 1152, whose weights a pair reads once, 243 / 194)
      const bool wide = static_cast<int64_t>(p.N) * p.K <= (48 << 20);   // (weights that stay in L2)
      const int short_k = wide && p.N >= 16384 ? 1152 : wide && p.N >= 9216 ? 1024 : p.N >= 6144 ? 768 : 384;
      const bool full = waves <= 3 && static_cast<int64_t>((p.M + 255) / 256) * ((p.N + 127) / 128) * 20 >= 17 * waves * ctx->num_sms;
      const bool f32 = cls == 6 && (waves == 1 || p.K <= short_k || (full && p.K <= 768 && cost <= 0.9 * pairs));
      if (f32 || (cls != 6 && cost <= pairs + spare + first)) return qdit_launch_gemm_t(ctx, A, W, p, a_unsigned, 256);
    }
    // (at most 128 rows: half of a pair's tokens would be padding; single CTAs / pairs: 1 x 193536 x 128 codes 18.8 / 44.4 us, 33 x 193536 x 384 22.5 / 42.7,
    // 100 x 65536 x 768 codes 14.9 / 19.0; from 129 rows on 160 x 193536 x 384 codes 63.7 / 46.2, 200 x 30720 x 3072 40 / 26.5)
    if (staged && p.M > BM && (slow ? pick_split(ctx, p.M, p.N, p.K, SPLIT_SPARE_SLOW) == 1 : !one_wave))
      return qdit_launch_gemm_pair(ctx, A, W, p, a_unsigned);
  }
  if (ctx->opt[QDIT_OPT_GEMM_BN] == 0) {
    const bool fast = cls >= 1 && cls <= 3 && !ctx->opt[QDIT_OPT_GEMM_GENERIC_EPILOGUE];
    const int split = pick_split(ctx, p.M, p.N, p.K, fast ? SPLIT_SPARE : SPLIT_SPARE_SLOW);
    if (split > 1) return qdit_launch_gemm_sk(ctx, A, W, p, a_unsigned, split, false);
  }
  switch (pick_bn(p.M, p.N, ctx->num_sms, ctx->opt[QDIT_OPT_GEMM_BN])) {
    case 64: return launch_gemm<64>(ctx, A, W, p, a_unsigned);
    case 128: return launch_gemm<128>(ctx, A, W, p, a_unsigned);
    default: return launch_gemm<192>(ctx, A, W, p, a_unsigned);
  }
}

extern "C" int32_t qdit_w8a8_linear(qdit_ctx* ctx, const void* A, const void* W, int64_t M, int64_t N, int64_t K,
                                    qdit_qparams a_qp, const float* a_scale_dev, uint32_t flags,
                                    const qdit_epilogue* epi, void* out, int64_t ldo) {
  return qdit_linear_impl(ctx, A, W, M, N, K, a_qp, a_scale_dev, flags, epi, out, ldo, false, nullptr, false, false, nullptr);
}

extern "C" int32_t qdit_w4a8_linear(qdit_ctx* ctx, const void* A, const void* W_packed, int64_t M, int64_t N, int64_t K,
                                    qdit_qparams a_qp, const float* a_scale_dev, uint32_t flags,
                                    const qdit_epilogue* epi, void* out, int64_t ldo, void* w8_scratch) {
  return qdit_linear_impl(ctx, A, W_packed, M, N, K, a_qp, a_scale_dev, flags, epi, out, ldo, true, w8_scratch, false, false, nullptr);
}
