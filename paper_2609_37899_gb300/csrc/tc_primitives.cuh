// tc_primitives.cuh -- thin inline-PTX wrappers for the sm_103a tensor-core
// path: shared-memory mbarriers (every wait bounded), 1-D bulk async copies,
// tensor-memory allocation, tcgen05.mma with shared-memory descriptors,
// tcgen05.commit and tcgen05.ld.
//
// Operand tiles use the canonical K-major layout without swizzle: an R x K
// fp16 tile is a grid of 8-row x 16-byte core matrices; element (r, k) sits
// at byte
//   (r / 8) * SBO + (k / 8) * LBO + (r % 8) * 16 + (k % 8) * 2
// with LBO = 128 (core matrices adjacent along K) and SBO = K * 16 (one
// 8-row group holds K / 8 core matrices).
#pragma once

#include <cstdint>
#include <cuda_fp16.h>

#include "soma_device.cuh"

namespace soma {
namespace tc {

// ---------------------------------------------------------------- smem ----
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// byte offset of element (r, k) inside a canonical K-major tile of K columns
__host__ __device__ __forceinline__ uint32_t kmajor_offset(int r, int k, int K) {
  return (uint32_t)((r >> 3) * (K * 16) + (k >> 3) * 128 + (r & 7) * 16 + (k & 7) * 2);
}

// --------------------------------------------------------------- mbarrier --
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}

__device__ __forceinline__ void mbar_fence_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}

// Suspend-time hint of one poll.  Measured on the gate kernel: with an
// explicit hint (any value from 1 to 500 ns) a launch takes 15% less time
// than with the default suspension, so waiting warps resume sooner.
constexpr uint32_t kSuspendHintNs = 100;

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n"
      " mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n"
      " selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity), "n"(kSuspendHintNs)
      : "memory");
  return ok != 0;
}

// Whether the phase with the given parity has completed, without waiting.
__device__ __forceinline__ bool mbar_test_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n"
      " mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Hint: bring the 128-byte line of a global address into L2.
__device__ __forceinline__ void prefetch_l2(const void* p) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

// Waits for the phase with the given parity to complete.  Gives up after
// `max_polls` unsuccessful polls (each try_wait suspends for at most about
// the hint) and returns false: no wait in this library can
// hang the GPU.  The caller records the timeout and skips the rest.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity,
                                          uint32_t max_polls = (1u << 22)) {
  for (uint32_t n = 0; n < max_polls; ++n)
    if (mbar_try_wait(bar, parity)) return true;
  return false;
}

// The kernels' waits.  One that runs out (`max_polls` polls) records the timeout
// and sets the CTA's abort flag; one that is still pending sees the flag within
// 64 polls and gives up too, so every warp leaves its loop.  A phase that is
// already complete costs one poll and no read of the flag.
//
// The calling lane's answer.  After an abort the lanes of a warp may get
// different ones: the caller votes before any lane leaves, for the others'
// shuffles, votes and tensor-memory instructions would wait for it without a
// bound.
__device__ __forceinline__ bool lane_wait_inline(uint64_t* bar, uint32_t parity,
                                                 volatile int* abort, int* status,
                                                 uint32_t max_polls = 1u << 22) {
  if (mbar_try_wait(bar, parity)) return true;
  for (uint32_t n = 1; n < max_polls; ++n) {
    if ((n & 63u) == 0 && *abort) return false;
    if (mbar_try_wait(bar, parity)) return true;
  }
  *abort = 1;
  atomicCAS(status, 0, kStatusTimeout);
  return false;
}

// The same with the polls after the first in a function of their own: in line
// they lengthen the loops of every role (SOMA N=8 step at T = 128: 20.4 ms, 21.8
// with them).
__device__ __noinline__ inline bool lane_wait_more(uint64_t* bar, uint32_t parity,
                                                   volatile int* abort, int* status,
                                                   uint32_t max_polls) {
  bool done = false;
  for (uint32_t n = 1; !done && n < max_polls; ++n) {
    if ((n & 63u) == 0 && *abort) return false;
    done = mbar_try_wait(bar, parity);
  }
  if (!done) {
    *abort = 1;
    atomicCAS(status, 0, kStatusTimeout);
  }
  return done;
}
__device__ __forceinline__ bool lane_wait(uint64_t* bar, uint32_t parity, volatile int* abort,
                                          int* status, uint32_t max_polls = 1u << 22) {
  return mbar_try_wait(bar, parity) || lane_wait_more(bar, parity, abort, status, max_polls);
}

// The whole warp's answer, the same in every lane: true once the phase has
// completed for all of them.
__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity, volatile int* abort,
                                          int* status, uint32_t max_polls = 1u << 22) {
  return __all_sync(0xffffffffu, lane_wait(bar, parity, abort, status, max_polls));
}

// ------------------------------------------------------------- bulk copy --
// 1-D async copy global -> shared completing on an mbarrier (tx bytes).
// Both addresses 16-byte aligned, size a multiple of 16.
__device__ __forceinline__ void bulk_g2s(void* smem_dst, const void* gmem_src, uint32_t bytes,
                                         uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
          "r"(smem_u32(smem_dst)),
      "l"(gmem_src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ void fence_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// ------------------------------------------------------------------ tmem --
// One warp allocates `ncols` (power of two, >= 32) tensor-memory columns and
// writes the base address to *slot (shared memory).
__device__ __forceinline__ void tmem_alloc(uint32_t* slot, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                   smem_u32(slot)),
               "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols)
               : "memory");
}

__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// ----------------------------------------------------------- descriptors --
// Shared-memory matrix descriptor: canonical K-major layout, no swizzle.
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);          // start address
  d |= (uint64_t)((lbo & 0x3FFFFu) >> 4) << 16;      // leading byte offset (along K)
  d |= (uint64_t)((sbo & 0x3FFFFu) >> 4) << 32;      // stride byte offset (8-row groups)
  d |= (uint64_t)1 << 46;                            // descriptor version for tcgen05
  // base offset 0, absolute LBO mode, layout type 0 = no swizzle
  return d;
}

// Instruction descriptor of kind::f16: fp16 A and B (K-major), fp32 D.
__host__ __device__ __forceinline__ uint32_t idesc_f16_f32(int M, int N) {
  uint32_t d = 0;
  d |= 1u << 4;                          // D format: f32
  d |= 0u << 7;                          // A format: f16
  d |= 0u << 10;                         // B format: f16
  d |= (uint32_t)(N >> 3) << 17;         // N / 8
  d |= (uint32_t)(M >> 4) << 24;         // M / 16
  return d;
}

// N of an instruction descriptor: the accumulator columns it writes.
__host__ __device__ __forceinline__ uint32_t idesc_columns(uint32_t idesc) {
  return ((idesc >> 17) & 0x3Fu) << 3;
}

// Descriptor split into its two 32-bit words: the low word holds the start
// address (bits 0..13, in 16-byte units) and LBO; moving a descriptor by a
// byte offset d that keeps the address below 256 KB is lo + (d >> 4).
// One thread of the (converged) warp: true in exactly one lane.
__device__ __forceinline__ bool elect_one() {
  uint32_t pred;
  asm volatile(
      "{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(pred));
  return pred != 0;
}

__device__ __forceinline__ void mma_f16_ss_lohi(uint32_t d_tmem, uint32_t a_lo, uint32_t a_hi,
                                                uint32_t b_lo, uint32_t b_hi, uint32_t idesc,
                                                uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n .reg .b64 da, db;\n setp.ne.b32 p, %6, 0;\n"
      " mov.b64 da, {%1, %2};\n mov.b64 db, {%3, %4};\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %5, p;\n}" ::"r"(d_tmem),
      "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(accumulate)
      : "memory");
}

// D[tmem] (+)= A[tmem] * B[smem]^T: A is 128 lanes (rows) x 8 columns, each
// 32-bit column holding the k pair (2c, 2c + 1) of fp16 values.
__device__ __forceinline__ void mma_f16_ts_lohi(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_lo,
                                                uint32_t b_hi, uint32_t idesc,
                                                uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n .reg .b64 db;\n setp.ne.b32 p, %5, 0;\n"
      " mov.b64 db, {%2, %3};\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], db, %4, p;\n}" ::"r"(d_tmem),
      "r"(a_tmem), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(accumulate)
      : "memory");
}

// 8 consecutive 32-bit columns of this thread's TMEM lane <- r[0..7].
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t* r) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(taddr),
               "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]),
               "r"(r[7])
               : "memory");
}

// 16 consecutive 32-bit columns of this thread's TMEM lane <- r[0..15].
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
      "%14,%15,%16};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
      "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}

__device__ __forceinline__ void tmem_wait_st() {
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// D[tmem] (+)= A[smem] * B[smem]^T  (M x N x 16), issued by one thread.
__device__ __forceinline__ void mma_f16_ss(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc,
                                           uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// Arrive on *bar once every previously issued tcgen05.mma of this thread
// has completed.
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
          smem_u32(bar))
      : "memory");
}

// 16 consecutive fp32 columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,"
      "%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]);
}

// 8 consecutive fp32 columns of this thread's TMEM lane, without waiting:
// the registers are valid after tmem_wait_ld().
__device__ __forceinline__ void tmem_ld8_nowait(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                 "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}

// 16x128b shape, one repetition: thread l receives column c + l % 4 of the
// lanes l / 4 and 8 + l / 4 of the 16-lane group at taddr (the lane field of
// taddr is the group's first lane).  Valid after tmem_wait_ld().
__device__ __forceinline__ void tmem_ld_16x128b(uint32_t taddr, uint32_t& r0, uint32_t& r1) {
  asm volatile("tcgen05.ld.sync.aligned.16x128b.x1.b32 {%0,%1}, [%2];"
               : "=r"(r0), "=r"(r1)
               : "r"(taddr));
}

// Two repetitions: (r0, r1) of columns c + l % 4 and (r2, r3) of columns c + 4 + l % 4.
__device__ __forceinline__ void tmem_ld_16x128b_x2(uint32_t taddr, uint32_t& r0, uint32_t& r1,
                                                   uint32_t& r2, uint32_t& r3) {
  asm volatile("tcgen05.ld.sync.aligned.16x128b.x2.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(taddr));
}

__device__ __forceinline__ void tmem_wait_ld() {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// 8 consecutive fp32 columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float* v) {
  uint32_t r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                 "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int j = 0; j < 8; ++j) v[j] = __uint_as_float(r[j]);
}

// Expands one raw probe word (parameter 2j of the run at bit j, parameter
// 2j+1 at bit j+16) into the fp16 pair word j of +-m values, m given as the
// doubled fp16 bit pattern mag2 = bits(m) * 0x10001: bit 1 <=> -m.  Element 2j
// lands in the low half (bit 15 = sign), 2j+1 in the high half.
template <int J>
__device__ __forceinline__ uint32_t pm_pair(uint32_t raw, uint32_t mag2) {
  static_assert(J >= 0 && J < 16, "pair index");
  return ((raw << (15 - J)) & 0x80008000u) | mag2;
}

// ----------------------------------------------------------- activations --
// 2^x and 1 / x by the special-function instructions, subnormals as zero, and
// exp(x) = 2^(x log2 e).  The sigmoids and softmax terms below add the power to
// a value of at least 1, where a power in the subnormal range is rounded away:
// over every float they equal the same forms with CUDA's __expf and __fdividef
// bit for bit (tests/test_gpu_activations.py).  An epilogue spends most of its
// time here: with those functions in their place the SOMA N=8 Adam step took
// 112.1 ms instead of 105.7, the N=256 step 172.8 instead of 161.9, the expert
// body's 580.9 instead of 570.7 (each with the kernels of that time).
__device__ __forceinline__ float ex2_ftz(float x) {
  float r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float rcp_ftz(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
constexpr float kLog2e = 1.4426950408889634f;  // exp(x) = 2^(x log2 e)

__device__ __forceinline__ float sigmoid_f(float x) {
  return rcp_ftz(1.0f + ex2_ftz(x * -kLog2e));
}
// tanh(x) = 2 sigmoid(2x) - 1
__device__ __forceinline__ float tanh_f(float x) {
  return fmaf(rcp_ftz(1.0f + ex2_ftz(x * (-2.0f * kLog2e))), 2.f, -1.f);
}
// h+- = o+- tanh(c+-) of the two signs as their sum and difference, from o and
// tanh(c) of each: the + product enters exactly, the - product rounded (one
// contraction of the two possible, written out so that every kernel has the
// same).
__device__ __forceinline__ void h_sum_diff(float op, float tp, float om, float tm, float& sum,
                                           float& dif) {
  const float hm = __fmul_rn(om, tm);
  sum = fmaf(op, tp, hm);
  dif = fmaf(op, tp, -hm);
}
// exp(x), x <= 0, for sums that hold a term of at least 1
__device__ __forceinline__ float exp_term(float x) { return ex2_ftz(x * kLog2e); }

// Gate tile rows: a 128-row tile covers 32 hidden units.  Tile row r lies in
// TMEM lane quarter r / 32 and holds gate (r / 8) % 4 of unit 8 (r / 32) +
// r % 8, so one quarter = 8 units x 4 gates, gate-major.  With this order a
// 16x128b tensor-memory load (rows l / 4 and 8 + l / 4 of a 16-lane half)
// gives thread l two gates of unit l / 4, and the two halves give all four.
__host__ __device__ __forceinline__ int tile_unit(int r) { return 8 * (r >> 5) + (r & 7); }
__host__ __device__ __forceinline__ int tile_gate(int r) { return (r >> 3) & 3; }

}  // namespace tc
}  // namespace soma
