// common.cuh -- shared device helpers of the FlashRelation kernels (sm_103a).
//
// Inline-PTX wrappers for mbarrier, TMA (cp.async.bulk.tensor), tcgen05 (TMEM
// allocation, MMA, commit, TMEM load/store, fences), the bounded pipeline wait with
// its abort protocol, and the small math helpers of the Relation role maps.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "relation.h"

namespace rel {

// ---------------------------------------------------------------------------
// Limits of the bounded waits.  A legitimate pipeline wait lasts microseconds; a
// wait that passes kWaitTimeoutNs is treated as a broken pipeline: the waiting
// thread records RELATION_ERR_TIMEOUT and the CTA unwinds (see Abort below).
// ---------------------------------------------------------------------------
constexpr unsigned long long kWaitTimeoutNs = 1000ull * 1000ull * 1000ull;  // 1 s

// Programmatic dependent launch (launch_pdl, kernels.h).  A kernel waits for the grids before it
// in the stream, complete and visible, before its first access to global memory and, where it has
// a set-up (barriers, TMEM), after that.  Without pdl_launch the next kernel's CTAs come in when
// every CTA of this one has ended; with it, once every CTA has called it.  Only the short
// elementwise kernels call it: in the tensor-core and fp32 tile kernels the next grid's waiting
// CTAs cost more than their early set-up gains (B 8, H 12, T 2048, d 64 forward + backward: 367 us
// with plain launches, 371 with pdl_launch everywhere, 356 as it is; B 2, H 8, T 1000, d 64 fp32:
// 335, 325, 320; B 4, H 8, T 4096, d 80 with the layer's transforms: 584, 603, 570; Linear
// Relation forward, B 1, H 12, T 32768: 159, 170, 150).
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait_and_launch() {
  pdl_wait();
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Compensated sum of a few floats: s the rounded sum, c the sum of the additions' errors.  Every
// product and sum whose rounding error is taken is rounded on its own (the _rn forms are never
// contracted to a multiply-add, which would round otherwise).
struct Sum2 {
  float s = 0.f, c = 0.f;
  __device__ __forceinline__ void add(float x) {
    const float t = __fadd_rn(s, x), z = __fsub_rn(t, s);
    c += __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(x, z));
    s = t;
  }
  // + f * log(x) for x > 0: x = 2^e y with y near 1, so that e ln 2 (ln 2 as a sum of two floats)
  // and log y, each with its rounding small against 1, take the place of one rounded logarithm
  __device__ __forceinline__ void add_log(float x, float f) {
    constexpr float kLn2 = 0.693147180559945309417f;
    constexpr float kLn2Lo = (float)(0.693147180559945309417 - (double)kLn2);
    int e;
    float y = frexpf(x, &e);
    if (y < 0.7071f) {
      y *= 2.f;
      --e;
    }
    const float a = __fmul_rn((float)e, kLn2), b = logf(y), fa = __fmul_rn(f, a), fb = __fmul_rn(f, b);
    add(fa);
    add(fb);
    c += fmaf(f, a, -fa) + fmaf(f, b, -fb) +
         f * fmaf((float)e, kLn2Lo, fmaf((float)e, kLn2, -a));
  }
};

__device__ __forceinline__ unsigned long long globaltimer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// ---------------------------------------------------------------------------
// mbarrier
// ---------------------------------------------------------------------------
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

// Non-blocking check of the phase with parity `parity` of `bar`.
__device__ __forceinline__ bool mbar_test_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

// Abort protocol: one int in shared memory.  A thread whose wait expires sets it and
// writes the status; every other bounded wait polls it and gives up as well, so each
// role leaves its loop and the CTA reaches its teardown (TMEM release) in bounded time.
struct Abort {
  volatile int* flag;  // shared memory
  int* dev_status;     // global, may be null
  __device__ __forceinline__ bool raised() const { return *flag != 0; }
  __device__ __forceinline__ void raise() const {
    *flag = 1;
    if (dev_status) atomicExch(dev_status, (int)RELATION_ERR_TIMEOUT);
  }
};

// Wait until the phase with parity `parity` of `bar` has completed.  Returns false
// (after raising the abort) when the wait exceeds kWaitTimeoutNs, or when another
// thread has raised the abort meanwhile.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, const Abort& ab,
                                          unsigned long long timeout_ns = kWaitTimeoutNs) {
  if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = globaltimer_ns();
  for (uint32_t it = 1;; ++it) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((it & 31u) == 0u) {
      if (ab.raised()) return false;
      if (globaltimer_ns() - t0 > timeout_ns) {
        ab.raise();
        return false;
      }
    }
  }
}

// Wait for two phases at once (phase pa of bar a, phase pb of bar b): b is checked first
// without blocking, so that its round trip overlaps the wait for a (b is usually complete
// long before).  Same bound and abort behaviour as mbar_wait.
__device__ __forceinline__ bool mbar_wait_both(uint32_t a, uint32_t pa, uint32_t b, uint32_t pb,
                                               const Abort& ab) {
  const bool db = mbar_test_wait(b, pb);
  const bool da = mbar_try_wait(a, pa);
  if (da && db) return true;
  if (!db && !mbar_wait(b, pb, ab)) return false;
  return da || mbar_wait(a, pa, ab);
}

// The bounded wait for a whole warp in warp-uniform code: true only when every lane saw
// the phase complete (a lane that timed out has raised the abort).
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, const Abort& ab) {
  return __all_sync(0xffffffffu, mbar_wait(bar, parity, ab));
}

// ---------------------------------------------------------------------------
// TMA (tensor maps are __grid_constant__ kernel parameters)
// ---------------------------------------------------------------------------
__device__ __forceinline__ void tma_prefetch_desc(const CUtensorMap* m) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(m)) : "memory");
}
// 4-D tiled load into shared memory, completing on `bar` (transaction bytes).
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* m, uint32_t bar,
                                            int c0, int c1, int c2, int c3) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4, %5, %6}], [%2];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(m)), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
      : "memory");
}
// 4-D tiled store from shared memory (bulk group); out-of-range rows are clipped.
__device__ __forceinline__ void tma_store_4d(const CUtensorMap* m, uint32_t src, int c0, int c1,
                                             int c2, int c3) {
  asm volatile(
      "cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%2, %3, %4, %5}], [%1];" ::"l"(
          reinterpret_cast<uint64_t>(m)),
      "r"(src), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
      : "memory");
}
__device__ __forceinline__ void tma_store_commit() {
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
// Wait until every committed bulk store / reduce has finished reading shared memory (its
// global writes may still be in flight; they complete before the kernel does).  Enough
// before a CTA releases or reuses the staging buffers.
__device__ __forceinline__ void tma_store_wait_read_all() {
  asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}
__device__ __forceinline__ void fence_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// ---------------------------------------------------------------------------
// tcgen05: tensor memory, MMA, commit, TMEM <-> registers
// ---------------------------------------------------------------------------
// Warp-collective.  Writes the TMEM base address of `ncols` columns into *dst_smem.
__device__ __forceinline__ void tmem_alloc(uint32_t dst_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem),
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
// D[tmem] (+)= A[smem desc] * B[smem desc]^T  (kind::f16, cta_group::1)
__device__ __forceinline__ void mma_ss(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc,
                                       uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// D[tmem] (+)= A[tmem] * B[smem desc]  (A operand read from tensor memory)
__device__ __forceinline__ void mma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc,
                                       uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
      "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// The same three instructions issued from warp-uniform code: every lane of the warp runs
// the surrounding loop and computes the (identical) descriptors, which then live in
// uniform registers, and elect.sync picks the one lane that issues.  From a divergent
// lane-0 branch the descriptors are per-thread values and each MMA costs ~67 cycles of
// issue at N = 64 against ~49 for the tensor core (measured on GB300).
__device__ __forceinline__ void mma_ss_w(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc,
                                         uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p, e;\n\t"
      "elect.sync _|e, 0xffffffff;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void mma_ts_w(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc,
                                         uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p, e;\n\t"
      "elect.sync _|e, 0xffffffff;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "@e tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
      "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Four k steps (K = 64) of one product under a single elect.sync: the operands advance by
// A_STEP and B_STEP (descriptor units of 16 bytes) a step; the first step accumulates if
// `accumulate`, the others always.
template <int A_STEP, int B_STEP>
__device__ __forceinline__ void mma_ss_w4(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc,
                                          uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p, e;\n\t.reg .b64 a1, a2, a3, b1, b2, b3;\n\t"
      "add.s64 a1, %1, %5;\n\tadd.s64 a2, %1, %6;\n\tadd.s64 a3, %1, %7;\n\t"
      "add.s64 b1, %2, %8;\n\tadd.s64 b2, %2, %9;\n\tadd.s64 b3, %2, %10;\n\t"
      "elect.sync _|e, 0xffffffff;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t"
      "setp.eq.b32 p, 0, 0;\n\t"
      "@e tcgen05.mma.cta_group::1.kind::f16 [%0], a1, b1, %3, p;\n\t"
      "@e tcgen05.mma.cta_group::1.kind::f16 [%0], a2, b2, %3, p;\n\t"
      "@e tcgen05.mma.cta_group::1.kind::f16 [%0], a3, b3, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "n"(A_STEP), "n"(2 * A_STEP),
      "n"(3 * A_STEP), "n"(B_STEP), "n"(2 * B_STEP), "n"(3 * B_STEP)
      : "memory");
}
// Two such products with A in tensor memory (steps 1 to 3 at columns A1, A2, A3 from the first)
// and, if COMMIT, the arrival on `bar` when they and everything issued before complete, under
// one elect.sync.
template <int A1, int A2, int A3, int B_STEP, bool COMMIT>
__device__ __forceinline__ void mma_ts_w4x2(uint32_t d0, uint32_t a0, uint64_t b0, uint32_t d1,
                                            uint32_t a1, uint64_t b1, uint32_t idesc,
                                            uint32_t accumulate, uint32_t bar) {
  asm volatile(
      "{\n\t.reg .pred p, t, e;\n\t.reg .b32 x1, x2, x3, y1, y2, y3;\n\t"
      ".reg .b64 u1, u2, u3, v1, v2, v3;\n\t"
      "add.s32 x1, %1, %9;\n\tadd.s32 x2, %1, %10;\n\tadd.s32 x3, %1, %11;\n\t"
      "add.s32 y1, %4, %9;\n\tadd.s32 y2, %4, %10;\n\tadd.s32 y3, %4, %11;\n\t"
      "add.s64 u1, %2, %12;\n\tadd.s64 u2, %2, %13;\n\tadd.s64 u3, %2, %14;\n\t"
      "add.s64 v1, %5, %12;\n\tadd.s64 v2, %5, %13;\n\tadd.s64 v3, %5, %14;\n\t"
      "elect.sync _|e, 0xffffffff;\n\t"
      "setp.ne.b32 p, %7, 0;\n\tsetp.eq.b32 t, 0, 0;\n\t"
      "@e tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %6, p;\n\t"
      "@e tcgen05.mma.cta_group::1.kind::f16 [%0], [x1], u1, %6, t;\n\t"
      "@e tcgen05.mma.cta_group::1.kind::f16 [%0], [x2], u2, %6, t;\n\t"
      "@e tcgen05.mma.cta_group::1.kind::f16 [%0], [x3], u3, %6, t;\n\t"
      "@e tcgen05.mma.cta_group::1.kind::f16 [%3], [%4], %5, %6, p;\n\t"
      "@e tcgen05.mma.cta_group::1.kind::f16 [%3], [y1], v1, %6, t;\n\t"
      "@e tcgen05.mma.cta_group::1.kind::f16 [%3], [y2], v2, %6, t;\n\t"
      "@e tcgen05.mma.cta_group::1.kind::f16 [%3], [y3], v3, %6, t;\n\t"
      "setp.ne.b32 p, %15, 0;\n\t"
      "and.pred e, e, p;\n\t"
      "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%8];\n\t}" ::"r"(
          d0),
      "r"(a0), "l"(b0), "r"(d1), "r"(a1), "l"(b1), "r"(idesc), "r"(accumulate), "r"(bar),
      "n"(A1), "n"(A2), "n"(A3), "n"(B_STEP), "n"(2 * B_STEP), "n"(3 * B_STEP),
      "n"(COMMIT ? 1 : 0)
      : "memory");
}
// Copy of a 128-row x 32-byte slice of a shared-memory matrix (the descriptor's layout,
// e.g. one K step of a 128-byte-swizzled K-major tile) into TMEM lanes 0-127, 8 columns:
// the A-operand layout of tcgen05.mma with A in TMEM.  Issued from warp-uniform code by one
// elected lane, in order with the MMAs of the same thread.
__device__ __forceinline__ void tmem_cp_w(uint32_t taddr, uint64_t s_desc) {
  asm volatile(
      "{\n\t.reg .pred e;\n\t"
      "elect.sync _|e, 0xffffffff;\n\t"
      "@e tcgen05.cp.cta_group::1.128x256b [%0], %1;\n\t}" ::"r"(taddr),
      "l"(s_desc)
      : "memory");
}
__device__ __forceinline__ void mma_commit_w(uint32_t bar) {
  asm volatile(
      "{\n\t.reg .pred e;\n\t"
      "elect.sync _|e, 0xffffffff;\n\t"
      "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(
          bar)
      : "memory");
}
// Arrive once on `bar` when every tcgen05 op issued so far by this thread completes.
__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
      : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_st_wait() {
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// 32 lanes x 32 bit, 16 consecutive columns: thread t of the warp receives the 16
// words of TMEM lane (lane_base + t).
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]),
        "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]),
        "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
      "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]),
      "r"(r[15])
      : "memory");
}

__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
      : "memory");
}

// Shared-memory matrix descriptor (tcgen05 "version 1" format):
//   bits  0-13 start address >> 4, 16-29 leading byte offset >> 4,
//   bits 32-45 stride byte offset >> 4, 46-47 version = 1, 49-51 base offset = 0,
//   bit  52 LBO mode = 0, 61-63 layout (2 = 128-byte swizzle).
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t saddr, uint32_t lbo_bytes,
                                                    uint32_t sbo_bytes) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
  d |= (uint64_t)((lbo_bytes >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo_bytes >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1u << 46;
  d |= (uint64_t)2u << 61;
  return d;
}

// Instruction descriptor of tcgen05.mma kind::f16 with bf16 A/B, fp32 D:
//   bits 4-5 D format (1 = f32), 7-9 A format (1 = bf16), 10-12 B format (1 = bf16),
//   bit 15 A major (0 = K-major, 1 = MN-major), bit 16 B major, 17-22 N >> 3,
//   24-28 M >> 4.
__host__ __device__ constexpr uint32_t idesc_bf16_f32(int M, int N, bool a_mn_major,
                                                      bool b_mn_major) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((a_mn_major ? 1u : 0u) << 15) |
         ((b_mn_major ? 1u : 0u) << 16) | ((uint32_t)(N >> 3) << 17) |
         ((uint32_t)(M >> 4) << 24);
}

// ---------------------------------------------------------------------------
// Work order of the tile kernels.  A unit is one 128-row tile of one head; unit w of the
// launch order maps to (t, bh) with t = 0 the head's heaviest tile.  The B * H heads are
// split into n_groups groups of equal size (the first BH % n_groups groups one head
// larger) taken one after the other, the heaviest tiles of a group's heads first, so that
// the rows the concurrently running units read and accumulate belong to few heads and
// stay in L2.  head_groups (kernels.h) keeps every group large enough that its work per
// resident CTA slot covers its heaviest unit; n_groups = 1 is plain heaviest-first order.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void grouped_unit(int w, int n_t, int BH, int n_groups, int& t,
                                             int& bh) {
  const int q = BH / n_groups, r = BH % n_groups;  // r groups of q + 1 heads, then q heads
  const int big = r * (q + 1) * n_t;
  int base, gs, rem;
  if (w < big) {
    const int g = w / ((q + 1) * n_t);
    base = g * (q + 1);
    gs = q + 1;
    rem = w - g * (q + 1) * n_t;
  } else {
    const int w2 = w - big;
    const int g = w2 / (q * n_t);
    base = r * (q + 1) + g * q;
    gs = q;
    rem = w2 - g * q * n_t;
  }
  t = rem / gs;
  bh = base + rem % gs;
}

// ---------------------------------------------------------------------------
// Math helpers
// ---------------------------------------------------------------------------
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float tanh_approx(float x) {
  float y;
  asm("tanh.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&h);
}

constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;

}  // namespace rel
