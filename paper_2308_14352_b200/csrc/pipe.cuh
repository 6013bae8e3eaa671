// mbarrier / TMA / bulk-copy wrappers shared by the pipelined expert kernels.  Every wait is
// bounded: a wait that runs out sets CHECK_WAIT_TIMEOUT in the context's check word, raises the
// CTA's abort flag and returns false, and the caller winds down without touching the stage.  The word behind the flag
// says whether the CTA still waits for the kernel in front (whose own waits are bounded): then waits go on but count no time.
#pragma once
#include "common.cuh"

namespace emoe {

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// The same test, but the hardware may park the thread until the phase completes or `ns` nanoseconds
// have passed: a waiting warp then costs neither issue slots nor shared-memory traffic, and it
// resumes as soon as the phase completes.
__device__ __forceinline__ bool mbar_try_wait_parked(uint32_t bar, uint32_t parity, uint32_t ns) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity), "r"(ns)
      : "memory");
  return ok != 0;
}
constexpr unsigned long long PIPE_WAIT_NS = 500000000ull;  // a wait gives up after half a second of its own
constexpr uint32_t PIPE_PARK_NS = 20000;                   // how long a waiting thread may be parked at a time
// The words of a CTA's waits, in shared memory: the first is the abort flag.
enum : int { PIPE_ABORT = 0, PIPE_FRONT = 1, PIPE_WORDS = 2 };
// The time a wait has had once the clock went from t0 to t1 over one poll: no more than twice what a poll may be parked
// for, so that a CTA that was switched out meanwhile does not take its absence for a wait that is stuck.
__host__ __device__ constexpr unsigned long long waited_ns(unsigned long long so_far, unsigned long long t0, unsigned long long t1, bool front) {
  return front ? 0 : so_far + (t1 - t0 < 2ull * PIPE_PARK_NS ? t1 - t0 : 2ull * PIPE_PARK_NS);
}
static_assert(waited_ns(0, 1000, 21000, false) == 20000 && waited_ns(70, 5, 5, false) == 70, "a poll counts what it took");
static_assert(waited_ns(0, 0, 10 * PIPE_WAIT_NS, false) < PIPE_WAIT_NS / 1000, "five seconds away are not five seconds of waiting");
static_assert(waited_ns(PIPE_WAIT_NS - 1, 1000, 21000, true) == 0, "the time of the kernel in front is not this one's");

// The rest of a wait whose first test failed.  Parked, not polled: the warps that feed a pipeline wait for most
// of its time, and their polling was a third of the instructions the SM executed.
static __device__ __noinline__ bool mbar_wait_parked(uint32_t bar, uint32_t parity, int* check_word, volatile int* abort_flag) {
  unsigned long long before, now, waited = 0;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(before));
  do {
    if (mbar_try_wait_parked(bar, parity, PIPE_PARK_NS)) return true;
    if (*abort_flag) return false;
    const bool front = abort_flag[PIPE_FRONT] != 0;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
    waited = waited_ns(waited, before, now, front);
    before = now;
  } while (waited < PIPE_WAIT_NS);
  *abort_flag = 1;
  atomicOr(check_word, CHECK_WAIT_TIMEOUT);
  return false;
}
// Bounded wait.  Returns false (after flagging the check word) if the phase never completed.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, int* check_word, volatile int* abort_flag) {
  return mbar_try_wait(bar, parity) || mbar_wait_parked(bar, parity, check_word, abort_flag);
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const void* tmap, int c0, int c1, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
      "l"(tmap), "r"(c0), "r"(c1), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}

// ... by a whole warp: a branch on one lane's answer may leave the lanes apart for as long as the compiler likes, and
// instructions that need the warp together (tcgen05.ld, tcgen05.st) may follow the wait
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, int* check_word, volatile int* abort_flag) {
  const bool done = mbar_try_wait(bar, parity);
  if (__all_sync(0xffffffffu, done)) return true;
  return __all_sync(0xffffffffu, done || mbar_wait_parked(bar, parity, check_word, abort_flag));
}

// ---- the same operations for a whole warp that runs convergent, one elected lane of which acts ----
// Tensor-core and TMA instructions take their operands from uniform registers.  In a branch that only one lane
// enters, every operand is moved there anew and each instruction of the loop costs its full latency
// (a loop of four MMAs, two waits and a commit took 850 cycles); a warp that stays together, with a
// warp index the compiler knows to be uniform, has them there already.
__device__ __forceinline__ int warp_uniform(int v) { return __shfl_sync(0xffffffffu, v, 0); }
__device__ __forceinline__ int uniform_warp() { return __shfl_sync(0xffffffffu, static_cast<int>(threadIdx.x) >> 5, 0); }
__device__ __forceinline__ uint32_t elect_one() {
  uint32_t on;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(on));
  return on;
}
__device__ __forceinline__ void mbar_arrive_if(uint32_t on, uint32_t bar, int count = 1) {
  asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %1, 0;\n\t@q mbarrier.arrive.shared::cta.b64 _, [%0], %2;\n\t}" ::"r"(bar), "r"(on),
               "r"(count)
               : "memory");
}
__device__ __forceinline__ void mbar_expect_tx_if(uint32_t on, uint32_t bar, uint32_t bytes) {
  asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %2, 0;\n\t@q mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n\t}" ::"r"(bar),
               "r"(bytes), "r"(on)
               : "memory");
}
__device__ __forceinline__ void tma_load_2d_if(uint32_t on, uint32_t dst, const void* tmap, int c0, int c1, uint32_t bar) {
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %5, 0;\n\t"
      "@q cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];\n\t}" ::"r"(dst),
      "l"(tmap), "r"(c0), "r"(c1), "r"(bar), "r"(on)
      : "memory");
}

}  // namespace emoe
