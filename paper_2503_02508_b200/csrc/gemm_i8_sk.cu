// W8A8 linear layer for few output tiles: the reduction is split over the CTAs of a cluster.
//
// What bounds it: a layer with few rows has fewer 128 x BN tiles than the chip has SMs (M = 256, N = 1152: 36 tiles of
// 128 x 64 on 148 SMs), and each CTA then reads its whole K alone at the 64 bytes per clock that one SM takes in (fc2 of
// DiT-XL/2: 864 KB, 7 of the 13 us the layer took).  Here S CTAs form a cluster, each multiplies its share of the
// k-blocks, and the int32 partial tiles meet in distributed shared memory: the tile's 16 groups of 8 rows are dealt out to
// the CTAs, each receives its groups of every partial tile, adds them (integers: exact in any order) and runs the fused
// epilogue on those rows, so the epilogue is split as well.
//
// Roles as in gemm_i8.cu (warp 0 TMA producer, warp 1 MMA issuer), one tile per cluster; the eight other warps move the
// accumulator to the CTAs that finish it (patches of 8 rows x 32 columns, 16-byte pieces XOR-swizzled by row) and, after the
// cluster barrier, finish one patch at a time.  With packed 4-bit weights (W4) the same eight warps, idle until the
// accumulator is complete, widen each weight stage in front of the tensor core (gemm_w4.cu has the layout): 256 x 1152 x 4608
// takes 8.5 us against 17.7 in the kernel that does this without splitting, 1 x 1152 x 4608 7.4 against 16.2, and
// 256 x 1152 x 1152 5.9 against 8.4.
#include "gemm_common.cuh"

namespace {

using namespace qgemm;

constexpr int SK_BN = 64;
constexpr int SK_EPI_WARPS = 8;
constexpr int SK_THREADS = 64 + SK_EPI_WARPS * 32;
constexpr int SK_CHUNKS = SK_BN / 32;
constexpr int PATCH_BYTES = 8 * 128;   // 8 rows x 32 int32

template <int S, bool W4>
struct SkCfg {
  static constexpr int GROUPS = (16 + S - 1) / S;               // row groups a CTA finishes, at most
  static constexpr int PATCHES = S * GROUPS * SK_CHUNKS;        // received: [source][group][chunk]
  // group g of 16 goes to CTA g * S / 16; CTA r has groups first(r) .. first(r + 1) - 1
  static __host__ __device__ constexpr int first(int r) { return (16 * r + S - 1) / S; }
  static constexpr int A_BYTES = BM * BK;
  static constexpr int B_BYTES = SK_BN * BK;
  static constexpr int P_BYTES = W4 ? SK_BN * BK / 2 : 0;       // packed weight tile
  static constexpr int STAGE_BYTES = A_BYTES + B_BYTES + P_BYTES;
  static constexpr int STAGES = W4 ? 6 : 7;
  static constexpr int BAR_BYTES = 256;
  static constexpr int TMEM_COLS = 64;
  static constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + PATCHES * PATCH_BYTES + BAR_BYTES + 1024;
};

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// address of the same shared-memory location in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}

template <int S, int EPI, bool W4>
__global__ void __launch_bounds__(SK_THREADS, 1)
gemm_i8_sk_kernel(const __grid_constant__ CUtensorMap tmap_a, const __grid_constant__ CUtensorMap tmap_w,
                  const GemmParams p, const uint32_t idesc) {
  using C = SkCfg<S, W4>;
  constexpr int STAGES = C::STAGES;
  extern __shared__ uint8_t smem_raw[];
  // identical layout in every CTA of the cluster: the alignment slack must not depend on the CTA
  uint8_t* smem = smem_raw + (1024u - (smem_u32(smem_raw) & 1023u)) % 1024u;
  uint8_t* sA = smem;
  uint8_t* sB = smem + STAGES * C::A_BYTES;
  uint8_t* sP = sB + STAGES * C::B_BYTES;
  uint8_t* patches = smem + STAGES * C::STAGE_BYTES;   // [source rank][row group][chunk]
  uint64_t* full_bar = reinterpret_cast<uint64_t*>(patches + C::PATCHES * PATCH_BYTES);
  uint64_t* empty_bar = full_bar + STAGES;
  uint64_t* ready_bar = empty_bar + STAGES;   // W4: weight tile widened (one arrival per warp)
  uint64_t* tfull_bar = ready_bar + STAGES;
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(tfull_bar + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_holder + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = static_cast<int>(cluster_rank());
  const int tile = blockIdx.x / S;
  const int m0 = (tile / p.num_n_tiles) * BM, n0 = (tile % p.num_n_tiles) * SK_BN;
  const int num_kb = (p.K + BK - 1) / BK;
  const int kb0 = num_kb * rank / S, kb1 = num_kb * (rank + 1) / S;   // S <= num_kb: never empty

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full_bar[s], 1);
      mbar_init(&empty_bar[s], 1);
      mbar_init(&ready_bar[s], SK_EPI_WARPS);
    }
    mbar_init(tfull_bar, 1);
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
  cluster_arrive();   // every CTA of the cluster has started: waited for before the first remote store
  const uint32_t tmem = *tmem_holder;   // (the roles that read what the previous kernel wrote wait for it themselves)

  // Work of this warp after the exchange: 8 rows x 32 columns at a time; what its first piece needs from global memory is asked for
  // before the products.
  const int g0 = C::first(rank), units = (C::first(rank + 1) - g0) * SK_CHUNKS;
  const int cg = lane & 3, rsub = lane >> 2;
  const uint32_t flags = epi_flags<EPI>(p);
  float a_scale = 0.0f, o_inv = 0.0f;
  ColParams cp;
  uint4 res = make_uint4(0u, 0u, 0u, 0u);
  auto locate = [&](int u, int& row, int& n) {
    row = m0 + (g0 + u / SK_CHUNKS) * 8 + rsub;
    n = n0 + (u % SK_CHUNKS) * 32 + cg * 8;
  };
  auto prefetch_columns = [&](int u) {
    int row, n;
    locate(u, row, n);
    if (row < p.M && n < p.N && !(flags & QDIT_EPI_OUT_I32)) load_col_params<EPI>(p, n, row / p.tokens, a_scale, cp);
  };
  auto prefetch_row = [&](int u) {
    int row, n;
    locate(u, row, n);
    if (row < p.M && n < p.N && (flags & QDIT_EPI_RESIDUAL)) res = *reinterpret_cast<const uint4*>(p.residual + static_cast<int64_t>(row) * p.ldo + n);
  };
  if (warp >= 2) {
    if (!p.early_params) grid_dependency_wait();
    a_scale = device_value(p.a_scale_dev, p.a_scale);
    if (flags & QDIT_EPI_QUANT_OUT) o_inv = __fdiv_rn(1.0f, device_value(p.o_scale_dev, p.o_scale));
    // (warps that widen weights first do not wait for the parameters in front of that)
    if ((!W4 || p.early_params) && warp - 2 < units) prefetch_columns(warp - 2);
    if (p.early_params) grid_dependency_wait();
    grid_dependency_release();
    if (warp - 2 < units) prefetch_row(warp - 2);
  }

  bool accumulated = false;
  const int quad = warp & 3, half = (warp - 2) >> 2;
  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    int stage = 0;
    uint32_t phase = 0;
    bool seen = true;   // the stage about to be filled is known to be free
    // the first stages' weights come while the previous kernel still runs
    const int ahead = !p.early ? 0 : kb1 - kb0 < STAGES ? kb1 - kb0 : STAGES;
    if (ahead > 0 && elect_one()) {
      for (int i = 0; i < ahead; ++i) {
        mbar_expect_tx(&full_bar[i], C::A_BYTES + (W4 ? C::P_BYTES : C::B_BYTES));
        if (W4) tma_load_2d(sP + i * C::P_BYTES, &tmap_w, (kb0 + i) * (BK / 2), n0, &full_bar[i]);
        else tma_load_2d(sB + i * C::B_BYTES, &tmap_w, (kb0 + i) * BK, n0, &full_bar[i]);
      }
    }
    __syncwarp();
    grid_dependency_wait();
    if (ahead > 0) {
      if (elect_one()) {
        for (int i = 0; i < ahead; ++i) tma_load_2d(sA + i * C::A_BYTES, &tmap_a, (kb0 + i) * BK, m0, &full_bar[i]);
      }
      __syncwarp();
      stage = ahead;
      if (stage == STAGES) { stage = 0; phase ^= 1u; seen = false; }
    }
    for (int kb = kb0 + ahead; kb < kb1; ++kb) {
      if (!mbar_wait_seen(seen, &empty_bar[stage], phase ^ 1u, abort_flag, p.status)) break;
      const bool wrap = stage + 1 == STAGES;
      seen = mbar_test_wait(&empty_bar[wrap ? 0 : stage + 1], phase ^ (wrap ? 0u : 1u));
      if (elect_one()) {
        mbar_expect_tx(&full_bar[stage], C::A_BYTES + (W4 ? C::P_BYTES : C::B_BYTES));
        tma_load_2d(sA + stage * C::A_BYTES, &tmap_a, kb * BK, m0, &full_bar[stage]);
        if (W4) tma_load_2d(sP + stage * C::P_BYTES, &tmap_w, kb * (BK / 2), n0, &full_bar[stage]);
        else tma_load_2d(sB + stage * C::B_BYTES, &tmap_w, kb * BK, n0, &full_bar[stage]);
      }
      __syncwarp();
      if (++stage == STAGES) { stage = 0; phase ^= 1u; }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    int stage = 0;
    uint32_t phase = 0;
    bool ok = true, seen = false;   // seen: the stage about to be multiplied is known to have landed
    uint64_t* const in_bar = W4 ? ready_bar : full_bar;
    for (int kb = kb0; kb < kb1; ++kb) {
      ok = mbar_wait_seen(seen, &in_bar[stage], phase, abort_flag, p.status);
      if (!ok) break;
      const bool wrap = stage + 1 == STAGES;
      seen = mbar_test_wait(&in_bar[wrap ? 0 : stage + 1], phase ^ (wrap ? 1u : 0u));
      tc_fence_after();
      const uint64_t a_desc = umma_desc_k_sw128(smem_u32(sA + stage * C::A_BYTES));
      const uint64_t b_desc = umma_desc_k_sw128(smem_u32(sB + stage * C::B_BYTES));
      if (elect_one()) {
#pragma unroll
        for (int k = 0; k < BK / UMMA_K; ++k)
          umma_i8(tmem, a_desc + static_cast<uint64_t>(k * (UMMA_K >> 4)), b_desc + static_cast<uint64_t>(k * (UMMA_K >> 4)), idesc,
                  (kb != kb0 || k != 0) ? 1u : 0u);
        umma_commit(&empty_bar[stage]);
      }
      __syncwarp();
      if (++stage == STAGES) { stage = 0; phase ^= 1u; }
    }
    if (ok && elect_one()) umma_commit(tfull_bar);
    __syncwarp();
  } else {
    bool ok = true;
    if constexpr (W4) {
      // 16-byte piece c of weight row n sits at n * 128 + ((c ^ (n & 7)) << 4) and comes from bytes 8 c .. of packed row n;
      // a thread widens piece ut & 7 of rows ut >> 3 and 32 + (ut >> 3)
      const int ut = (warp - 2) * 32 + lane, row = ut >> 3, c = ut & 7;
      int stage = 0;
      uint32_t phase = 0;
      for (int kb = kb0; kb < kb1 && ok; ++kb) {
        ok = mbar_wait_warp(&full_bar[stage], phase, abort_flag, p.status);
        if (!ok) break;
        const uint8_t* src = sP + stage * C::P_BYTES + row * 64 + c * 8;
        uint8_t* dst = sB + stage * C::B_BYTES + row * 128 + ((c ^ (row & 7)) << 4);
        const uint2 a = *reinterpret_cast<const uint2*>(src), b = *reinterpret_cast<const uint2*>(src + 32 * 64);
        *reinterpret_cast<uint4*>(dst) = widen_w4x16(a);
        *reinterpret_cast<uint4*>(dst + 32 * 128) = widen_w4x16(b);
        fence_async_smem();   // the tensor core reads the stage through the async proxy
        __syncwarp();
        if (lane == 0) mbar_arrive(&ready_bar[stage]);
        if (++stage == STAGES) { stage = 0; phase ^= 1u; }
      }
    }
    if (W4 && !p.early_params && warp - 2 < units) prefetch_columns(warp - 2);
    accumulated = ok && mbar_wait_warp(tfull_bar, 0, abort_flag, p.status);
  }
  cluster_wait();
  if (accumulated) {
    // ------------------------------------------------------------------ the partial tile to the CTAs that finish it
    tc_fence_after();
    const int group = quad * 4 + (lane >> 3), dest = group * S / 16;   // of this thread's row
#pragma unroll 1
    for (int c = half; c < SK_CHUNKS; c += SK_EPI_WARPS / 4) {
      uint32_t v[32];
      tmem_ld_32x32(tmem + (static_cast<uint32_t>(quad * 32) << 16) + static_cast<uint32_t>(c * 32), v);
      tmem_ld_wait();
      const uint32_t patch = map_rank(smem_u32(patches + ((rank * C::GROUPS + group - C::first(dest)) * SK_CHUNKS + c) * PATCH_BYTES),
                                      static_cast<uint32_t>(dest));
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const uint32_t addr = patch + static_cast<uint32_t>((lane & 7) * 128 + ((j ^ (lane & 7)) << 4));
        asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v[4 * j]), "r"(v[4 * j + 1]),
                     "r"(v[4 * j + 2]), "r"(v[4 * j + 3])
                     : "memory");
      }
    }
    tc_fence_before();
  }
  cluster_arrive();
  cluster_wait();
  if (warp >= 2 && !*abort_flag) {
    float top = 0.0f;
#pragma unroll 1
    for (int u = warp - 2; u < units; u += SK_EPI_WARPS) {
      if (u != warp - 2) {
        prefetch_columns(u);
        prefetch_row(u);
      }
      int row, n;
      locate(u, row, n);
      uint4 lo = make_uint4(0u, 0u, 0u, 0u), hi = lo;
#pragma unroll
      for (int s = 0; s < S; ++s) {
        const uint8_t* patch = patches + (s * C::GROUPS * SK_CHUNKS + u) * PATCH_BYTES + rsub * 128;
        const uint4 l = *reinterpret_cast<const uint4*>(patch + (((2 * cg) ^ rsub) << 4));
        const uint4 h = *reinterpret_cast<const uint4*>(patch + (((2 * cg + 1) ^ rsub) << 4));
        lo.x += l.x; lo.y += l.y; lo.z += l.z; lo.w += l.w;
        hi.x += h.x; hi.y += h.y; hi.z += h.z; hi.w += h.w;
      }
      if (row < p.M && n < p.N) epilogue8<EPI>(p, lo, hi, cp, res, row, n, o_inv, top);
    }
    __syncwarp();
    if (EPI == 7) publish_absmax(p.absmax, top);
  }
  if (*abort_flag && warp == 0) {
    for (int i = 0; i < 2000; ++i) __nanosleep(1000);  // let copies in flight land before shared memory goes away
  }
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, C::TMEM_COLS);
  }
}

template <int S, int EPI, bool W4>
int32_t launch_sk_epi(qdit_ctx* ctx, const void* A, const void* W, GemmParams& p, bool a_unsigned) {
  using C = SkCfg<S, W4>;
  QDIT_TRY(qdit_allow_smem(ctx, gemm_i8_sk_kernel<S, EPI, W4>, C::SMEM_BYTES));
  CUtensorMap ta, tw;
  QDIT_TRY(qdit_get_tmap(ctx, A, p.M, p.K, p.K, BM, BK, 1, 1, &ta));
  if (W4) QDIT_TRY(qdit_get_tmap(ctx, W, p.N, p.K / 2, p.K / 2, SK_BN, BK / 2, 0, 1, &tw));
  else QDIT_TRY(qdit_get_tmap(ctx, W, p.N, p.K, p.K, SK_BN, BK, 1, 1, &tw));
  p.num_m_tiles = (p.M + BM - 1) / BM;
  p.num_n_tiles = (p.N + SK_BN - 1) / SK_BN;
  const uint32_t idesc = umma_idesc_i8(BM, SK_BN, a_unsigned);
  ProfScope prof(ctx, QDIT_PROF_GEMM, 2.0 * p.M * static_cast<double>(p.N) * p.K);
  QDIT_CUDA_CHECK(ctx, qdit_launch_cluster(ctx, gemm_i8_sk_kernel<S, EPI, W4>, dim3(p.num_m_tiles * p.num_n_tiles * S), dim3(SK_THREADS), C::SMEM_BYTES, S,
                                           ta, tw, p, idesc));
  return qdit_after_launch(ctx, "gemm_i8_sk_kernel");
}

template <int S, bool W4>
int32_t launch_sk(qdit_ctx* ctx, const void* A, const void* W, GemmParams& p, bool a_unsigned) {
  switch (epi_token_major(p, ctx->opt[QDIT_OPT_GEMM_GENERIC_EPILOGUE] != 0)) {
    case 1: return launch_sk_epi<S, 1, W4>(ctx, A, W, p, a_unsigned);
    case 2: return launch_sk_epi<S, 2, W4>(ctx, A, W, p, a_unsigned);
    case 3: return launch_sk_epi<S, 3, W4>(ctx, A, W, p, a_unsigned);
    case 7: return launch_sk_epi<S, 7, W4>(ctx, A, W, p, a_unsigned);
    default: return launch_sk_epi<S, 0, W4>(ctx, A, W, p, a_unsigned);
  }
}

}  // namespace

int32_t qdit_launch_gemm_sk(qdit_ctx* ctx, const void* A, const void* W, qgemm::GemmParams& p, bool a_unsigned, int split, bool packed4) {
  switch (split) {
    case 6: return packed4 ? launch_sk<6, true>(ctx, A, W, p, a_unsigned) : launch_sk<6, false>(ctx, A, W, p, a_unsigned);
    case 4: return packed4 ? launch_sk<4, true>(ctx, A, W, p, a_unsigned) : launch_sk<4, false>(ctx, A, W, p, a_unsigned);
    case 3: return packed4 ? launch_sk<3, true>(ctx, A, W, p, a_unsigned) : launch_sk<3, false>(ctx, A, W, p, a_unsigned);
    default: return packed4 ? launch_sk<2, true>(ctx, A, W, p, a_unsigned) : launch_sk<2, false>(ctx, A, W, p, a_unsigned);
  }
}

// Asked once per context and cluster size (the answer depends on the device's layout of SMs only: a CTA takes a whole SM).
template <int S>
static int sk_clusters(qdit_ctx* ctx) {
  using C = SkCfg<S, false>;
  if (qdit_allow_smem(ctx, gemm_i8_sk_kernel<S, 0, false>, C::SMEM_BYTES) != QDIT_OK) return 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(S);
  cfg.blockDim = dim3(SK_THREADS);
  cfg.dynamicSmemBytes = C::SMEM_BYTES;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = S;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, gemm_i8_sk_kernel<S, 0, false>, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}
int qdit_gemm_sk_clusters(qdit_ctx* ctx, int split) {
  int& n = ctx->sk_clusters[split];
  if (n == 0) {
    n = split == 6 ? sk_clusters<6>(ctx) : split == 4 ? sk_clusters<4>(ctx) : split == 3 ? sk_clusters<3>(ctx) : sk_clusters<2>(ctx);
    if (n == 0) n = -1;
  }
  return n;
}
