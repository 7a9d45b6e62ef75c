// Device-side helpers: PTX wrappers for mbarrier, TMA, tcgen05/TMEM, plus small numeric utilities.
// sm_100a only.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace qd {

// ----------------------------------------------------------------------------- addresses
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// One thread of the (converged) warp, the same one at every call.  The compiler knows that a branch on the result holds a
// single thread, so operands of the tensor-core and copy instructions inside it (descriptors, addresses) stay in uniform
// registers; behind `lane == 0` it moves every operand there before each instruction.
__device__ __forceinline__ bool elect_one() {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "elect.sync _|p, 0xffffffff;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok));
  return ok != 0;
}

// ----------------------------------------------------------------------------- mbarrier
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_fence_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// Arrive without memory ordering: used where the barrier only hands back tensor memory (ordered by the
// tcgen05 fences) and must not wait for the thread's outstanding global stores to become visible.
__device__ __forceinline__ void mbar_arrive_relaxed(uint64_t* bar) {
  asm volatile("mbarrier.arrive.relaxed.cta.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// Programmatic dependent launch.  A kernel launched with the programmatic-stream-serialization attribute may
// begin (CTA scheduling, barrier set-up, tensor-memory allocation, descriptor prefetch) while the kernel
// before it in the stream is still running.  grid_dependency_wait() returns once that kernel has completed
// and its writes are visible; nothing before it may touch global memory that another kernel writes or reads.
// grid_dependency_release() lets the NEXT kernel of the stream start its own preamble.  Both are no-ops for
// a kernel launched without the attribute.
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_dependency_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// A quantizer's scale: the one in device memory, if there is one.  (Not through the read-only path: the launch in front may write it while
// this kernel is already resident.)
__device__ __forceinline__ float device_value(const float* dev, float value) {
  return dev ? *dev : value;
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// One look at the barrier, without waiting.
__device__ __forceinline__ bool mbar_test_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Bounded wait: polls the barrier at most kSpinLimit times.  On expiry it raises the CTA's abort flag
// (shared) and the device status word (global) and returns false; it also returns false as soon as
// another thread of the CTA has raised the abort flag, so every role drains to the common exit.
constexpr uint32_t kSpinLimit = 1u << 24;
__device__ __forceinline__ bool mbar_wait_limited(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int* status,
                                                  uint32_t limit) {
  for (uint32_t i = 0; i < limit; ++i) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((i & 63u) == 63u && *abort_flag) return false;
  }
  *abort_flag = 1;
  atomicExch(status, 1);
  return false;
}
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int* status) {
  return mbar_wait_limited(bar, parity, abort_flag, status, kSpinLimit);
}

// The same for a whole converged warp: every lane gets the same answer, so the warp stays together on a time-out too.
__device__ __forceinline__ bool mbar_wait_warp(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int* status) {
  return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag, status));
}

// The same for a wait that other warps' work hangs on: it looks again and again.  try_wait may suspend the thread, and beside warps that
// keep the special-function unit busy the return from it took 300-500 clocks, a look that succeeds 180-250.  (For long waits
// that nobody else waits behind, try_wait is the better one: the looks take slots of the queue that everything else goes through.)
// Bounded in the same way: at most `limit` looks, in steps of 1024.
constexpr uint32_t kPollLimit = 1u << 27;
__device__ __forceinline__ bool mbar_poll_warp(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int* status, uint32_t limit = kPollLimit) {
  bool ok = true;
  for (uint32_t i = 1; !mbar_test_wait(bar, parity); ++i) {
    if ((i & 1023u) == 0u && (i >= limit || *abort_flag)) {
      ok = false;
      break;
    }
  }
  ok = __all_sync(0xffffffffu, ok);
  if (!ok && *abort_flag == 0) {
    *abort_flag = 1;
    atomicExch(status, 1);
  }
  return ok;
}
__device__ __forceinline__ bool mbar_poll_seen(bool seen, uint64_t* bar, uint32_t parity, volatile int* abort_flag, int* status) {
  return __all_sync(0xffffffffu, seen) || mbar_poll_warp(bar, parity, abort_flag, status);
}

// The same behind an earlier mbar_test_wait of the same phase.  A look at a barrier takes about 200 clocks in these
// kernels; a role that looks at its next barrier before it issues the work of the current one does not wait for that.
__device__ __forceinline__ bool mbar_wait_seen(bool seen, uint64_t* bar, uint32_t parity, volatile int* abort_flag, int* status) {
  return __all_sync(0xffffffffu, seen) || mbar_wait_warp(bar, parity, abort_flag, status);
}

// For a role whose wait for a copy ran out, or that left through the abort flag: the copies still in flight get 2 ms (a copy takes
// microseconds) to land before the CTA's shared memory is released.  Their barriers are of no use here: a wait returns at once when the
// flag is up.
__device__ __forceinline__ void leave_time_for_copies() {
  for (int i = 0; i < 2000; ++i) __nanosleep(1000);
}

// ----------------------------------------------------------------------------- TMA (every copy serves the issuing CTA alone)
__device__ __forceinline__ void tma_prefetch_desc(const void* tmap) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(tmap)) : "memory");
}
// 2-D tiled load global -> shared of the calling CTA; c0 = innermost (column) coordinate, c1 = row.
__device__ __forceinline__ void tma_load_2d(void* smem_dst, const void* tmap, int32_t c0, int32_t c1, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
      ::"r"(smem_u32(smem_dst)), "l"(reinterpret_cast<uint64_t>(tmap)), "r"(c0), "r"(c1), "r"(smem_u32(bar))
      : "memory");
}

// 2-D tiled store shared -> global (bulk async group of the issuing thread).  Rows or columns of the box that
// fall outside the tensor are not written.  c0 (innermost coordinate) times the element size must be a
// multiple of 16 bytes.
__device__ __forceinline__ void tma_store_2d(const void* tmap, const void* smem_src, int32_t c0, int32_t c1) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];"
               ::"l"(reinterpret_cast<uint64_t>(tmap)), "r"(c0), "r"(c1), "r"(smem_u32(smem_src))
               : "memory");
}
__device__ __forceinline__ void tma_store_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// Waits until at most N of this thread's bulk groups have not yet finished READING their shared-memory source.
template <int N>
__device__ __forceinline__ void tma_store_wait_read() { asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory"); }
// Waits until all of this thread's bulk groups have completed (their global writes included).
__device__ __forceinline__ void tma_store_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// Makes generic-proxy writes to shared memory visible to the async proxy (TMA, tensor-core operand reads).
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// ----------------------------------------------------------------------------- tcgen05 / TMEM
__device__ __forceinline__ void tmem_alloc(uint32_t* smem_holder, uint32_t ncols) {  // whole warp
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(smem_holder)),
               "r"(ncols)
               : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {  // whole warp
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// D[tmem] (+)= A[smem desc] * B[smem desc], 8-bit integer operands, int32 accumulate.  One thread issues.
__device__ __forceinline__ void umma_i8(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                        uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Arrives on `bar` once every tcgen05 operation this thread issued so far has completed.
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}
// 32 lanes x 32 consecutive 32-bit columns: thread i of the warp gets lane (base_lane + i), v[j] = column j.
__device__ __forceinline__ void tmem_ld_32x32(uint32_t taddr, uint32_t (&v)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]),
        "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
        "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
// The same wait, tied to the registers of a load that is still in flight: nothing that reads them can be moved before it.
__device__ __forceinline__ void tmem_ld_wait_for(uint32_t (&v)[32]) {
  asm volatile(
      "tcgen05.wait::ld.sync.aligned;"
      : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]), "+r"(v[8]),
        "+r"(v[9]), "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15]), "+r"(v[16]),
        "+r"(v[17]), "+r"(v[18]), "+r"(v[19]), "+r"(v[20]), "+r"(v[21]), "+r"(v[22]), "+r"(v[23]), "+r"(v[24]),
        "+r"(v[25]), "+r"(v[26]), "+r"(v[27]), "+r"(v[28]), "+r"(v[29]), "+r"(v[30]), "+r"(v[31])
      :
      : "memory");
}
// 16 lanes x 32 consecutive 32-bit columns in the layout of a matrix-multiply accumulator fragment: thread t of the
// warp gets, for column block b = 0..3,  v[4b], v[4b+1] = lane (base_lane + t/4), columns 8b + 2(t%4), + 1
//                                        v[4b+2], v[4b+3] = lane (base_lane + t/4 + 8), the same columns.
__device__ __forceinline__ void tmem_ld_16x256b_x4(uint32_t taddr, uint32_t (&v)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x4.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
      : "r"(taddr)
      : "memory");
}
// Four 8 x 8 matrices of 16-bit elements between registers and shared memory, transposed: thread t holds, of
// matrix j (register j), the elements (rows 2(t%4), 2(t%4) + 1; column t/4), low half = the even row; thread t
// supplies the address of row t%8 of matrix t/8 (16 bytes per row).
__device__ __forceinline__ void stmatrix_x4_trans(uint32_t addr, uint32_t r0, uint32_t r1, uint32_t r2, uint32_t r3) {
  asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(r0), "r"(r1),
               "r"(r2), "r"(r3)
               : "memory");
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(addr)
               : "memory");
}

// Shared-memory matrix descriptor for a K-major operand tile staged by TMA with 128-byte swizzle:
// rows are 128 bytes, groups of 8 rows are 1024 bytes apart, tile base 1024-byte aligned.
__device__ __forceinline__ uint64_t umma_desc_k_sw128(uint32_t smem_addr) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((smem_addr & 0x3FFFFu) >> 4);  // start address
  d |= static_cast<uint64_t>(1) << 16;                      // leading byte offset (unused with swizzle)
  d |= static_cast<uint64_t>(1024 >> 4) << 32;              // stride byte offset: 8-row group pitch
  d |= static_cast<uint64_t>(1) << 46;                      // descriptor version of this architecture
  d |= static_cast<uint64_t>(2) << 61;                      // 128-byte swizzle
  return d;
}

// Generic shared-memory matrix descriptor: layout 2 = 128-byte swizzle, 6 = 32-byte swizzle; sbo = byte
// distance between 8-row groups (rows along MN for a K-major operand, along K for an MN-major one).
__device__ __forceinline__ uint64_t umma_desc(uint32_t smem_addr, uint32_t sbo, uint32_t layout) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((smem_addr & 0x3FFFFu) >> 4);
  d |= static_cast<uint64_t>(1) << 16;
  d |= static_cast<uint64_t>((sbo >> 4) & 0x3FFF) << 32;
  d |= static_cast<uint64_t>(1) << 46;
  d |= static_cast<uint64_t>(layout) << 61;
  return d;
}
// Instruction descriptor for kind::f16 with bf16 operands and f32 accumulator; b_mn: B operand is MN-major
// (its N index is the contiguous one in shared memory).
__host__ __device__ constexpr uint32_t umma_idesc_bf16(uint32_t M, uint32_t N, bool b_mn) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((b_mn ? 1u : 0u) << 16) | ((N >> 3) << 17) | ((M >> 4) << 24);
}
__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                          uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// D[tmem] (+)= A[tmem] * B[smem desc]: the A operand (M = 128 rows on the lanes, 16 bf16 per instruction along K)
// is read from tensor memory, where a 32-bit column holds two consecutive K elements of a row (low half first).
__device__ __forceinline__ void umma_bf16_ta(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                             uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// 32 lanes x 16 consecutive 32-bit columns from registers: thread i of the warp writes lane (base_lane + i).
__device__ __forceinline__ void tmem_st_32x16(uint32_t taddr, const uint32_t (&v)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
      ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]),
        "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
      : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_ld_32x16(uint32_t taddr, uint32_t (&v)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_ld_32x8(uint32_t taddr, uint32_t (&v)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
               : "r"(taddr)
               : "memory");
}
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Instruction descriptor for kind::i8: int32 accumulator, A signed or unsigned bytes, B signed bytes,
// both K-major, tile M x N.
__host__ __device__ constexpr uint32_t umma_idesc_i8(uint32_t M, uint32_t N, bool a_unsigned) {
  return (2u << 4)                        // D format: S32
         | ((a_unsigned ? 0u : 1u) << 7)  // A format: 0 = U8, 1 = S8
         | (1u << 10)                     // B format: S8
         | ((N >> 3) << 17) | ((M >> 4) << 24);
}

// ----------------------------------------------------------------------------- numerics
__device__ __forceinline__ float quantize_code(float x, float inv_scale, float zp, float qmin, float qmax) {
  // Eq. 1 in float32: one rounded product, nearest-even, then zero-point and clip.
  float r = rintf(__fmul_rn(x, inv_scale));
  return fminf(fmaxf(r + zp, qmin), qmax);
}
// Same decision as quantize_code, as an integer and without conversion instructions: adding 1.5 * 2^23
// rounds a float of magnitude < 2^22 to the nearest integer (ties to even) and leaves that integer in the
// low mantissa bits.  The product is clamped to +-1024 first, which cannot change the clipped code.
__device__ __forceinline__ int quantize_code_i(float x, float inv_scale, int zp, int qmin, int qmax) {
  const float t = fminf(fmaxf(__fmul_rn(x, inv_scale), -1024.0f), 1024.0f);
  const int r = __float_as_int(__fadd_rn(t, 12582912.0f)) - 0x4B400000;
  return min(max(r + zp, qmin), qmax);
}
__device__ __forceinline__ float gelu_tanh_f(float x) {
  // 0.5 x (1 + tanh(u)) = x / (1 + exp(-2u)),  u = sqrt(2/pi) (x + 0.044715 x^3)
  //                     = x / (1 + 2^(x (a + b x^2))),  a = -2 sqrt(2/pi) log2(e),  b = 0.044715 a
  // (7 instructions, two of them on the special-function unit)
  const float a = -2.3022081998f, b = -0.1029432396f;
  const float e = ex2_approx(x * fmaf(x * x, b, a));
  return __fdividef(x, 1.0f + e);
}
__device__ __forceinline__ float silu_f(float x) { return x / (1.0f + expf(-x)); }

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// Folds a warp's largest magnitude (of non-negative values per lane) into *slot, which holds 0 or an earlier one.
__device__ __forceinline__ void publish_absmax(float* slot, float m) {
  m = warp_max(m);
  if ((threadIdx.x & 31) == 0) atomicMax(reinterpret_cast<int*>(slot), __float_as_int(m));
}

__device__ __forceinline__ void unpack_bf16x2(uint32_t w, float& a, float& b) {
  a = __uint_as_float(w << 16);
  b = __uint_as_float(w & 0xFFFF0000u);
}
__device__ __forceinline__ uint32_t pack_bf16x2(float a, float b) {
  __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&h);
}

// 8 consecutive values from 16-byte aligned memory, widened to float.
template <typename T>
struct Load8;
template <>
struct Load8<__nv_bfloat16> {
  static __device__ __forceinline__ void load(const __nv_bfloat16* p, float (&v)[8]) {
    const uint4 w = *reinterpret_cast<const uint4*>(p);
    unpack_bf16x2(w.x, v[0], v[1]);
    unpack_bf16x2(w.y, v[2], v[3]);
    unpack_bf16x2(w.z, v[4], v[5]);
    unpack_bf16x2(w.w, v[6], v[7]);
  }
};
template <>
struct Load8<float> {
  static __device__ __forceinline__ void load(const float* p, float (&v)[8]) {
    const float4 a = *reinterpret_cast<const float4*>(p);
    const float4 b = *reinterpret_cast<const float4*>(p + 4);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
  }
};

// 8 integral code values in [-128, 255] -> 8 stored bytes (low byte of the integer).
__device__ __forceinline__ uint2 pack_codes8(const float (&c)[8]) {
  uint32_t lo = 0, hi = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    lo |= (static_cast<uint32_t>(__float2int_rn(c[i])) & 0xFFu) << (8 * i);
    hi |= (static_cast<uint32_t>(__float2int_rn(c[4 + i])) & 0xFFu) << (8 * i);
  }
  return make_uint2(lo, hi);
}
// 8 integer codes in [-128, 255] -> 8 stored bytes.
__device__ __forceinline__ uint2 pack_codes8_i(const int (&c)[8]) {
  uint32_t lo = 0, hi = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    lo |= (static_cast<uint32_t>(c[i]) & 0xFFu) << (8 * i);
    hi |= (static_cast<uint32_t>(c[4 + i]) & 0xFFu) << (8 * i);
  }
  return make_uint2(lo, hi);
}
// Eq. 1 for 8 values straight to 8 stored bytes, without conversion instructions:
// clip(rne(t) + z, qmin, qmax) == rne(clamp(t, qmin - z, qmax - z)) + z because the bounds are integers, and
// adding 1.5 * 2^23 to a float of magnitude < 2^22 rounds it to the nearest integer (ties to even) and
// leaves that integer in the low mantissa bits.  Same codes as quantize_code for every input (NaN -> qmin).
// quantize_pack8_scaled takes t = x / s already formed.
__device__ __forceinline__ uint2 quantize_pack8_scaled(const float (&t)[8], float zp, float qmin, float qmax) {
  const float lo_f = qmin - zp, hi_f = qmax - zp;
  const int z = static_cast<int>(zp);
  uint32_t m[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float c = fminf(fmaxf(t[i], lo_f), hi_f);
    m[i] = static_cast<uint32_t>(__float_as_int(__fadd_rn(c, 12582912.0f)));
  }
  if (z != 0) {  // uniform over the grid: symmetric quantizers skip the eight adds
#pragma unroll
    for (int i = 0; i < 8; ++i) m[i] += static_cast<uint32_t>(z);
  }
  uint2 r;
  r.x = __byte_perm(__byte_perm(m[0], m[1], 0x0040), __byte_perm(m[2], m[3], 0x0040), 0x5410);
  r.y = __byte_perm(__byte_perm(m[4], m[5], 0x0040), __byte_perm(m[6], m[7], 0x0040), 0x5410);
  return r;
}
__device__ __forceinline__ uint2 quantize_pack8(const float (&x)[8], float inv_scale, float zp, float qmin, float qmax) {
  float t[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) t[i] = __fmul_rn(x[i], inv_scale);
  return quantize_pack8_scaled(t, zp, qmin, qmax);
}
__device__ __forceinline__ uint4 pack_bf16x8(const float (&y)[8]) {
  return make_uint4(pack_bf16x2(y[0], y[1]), pack_bf16x2(y[2], y[3]), pack_bf16x2(y[4], y[5]), pack_bf16x2(y[6], y[7]));
}

}  // namespace qd
