// Device helpers of the tensor-core kernels: bounded mbarrier waits, tcgen05 MMA
// issue, commit and fences (inline PTX, sm_103a).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

namespace dmrg {
namespace {

constexpr long long WAIT_CYCLES = 3000000000LL; // about 1.5 s at 2 GHz (fits the 32-bit clock)

__device__ __forceinline__ uint32_t saddr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint32_t a, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(a), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t a) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(a) : "memory");
}

// one try that may sleep up to about `ns` nanoseconds until the phase completes
__device__ __forceinline__ bool mbar_try_ns(uint32_t a, uint32_t parity, uint32_t ns) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(ok)
      : "r"(a), "r"(parity), "r"(ns)
      : "memory");
  return ok != 0;
}

__device__ __forceinline__ bool mbar_try(uint32_t a, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(ok)
      : "r"(a), "r"(parity)
      : "memory");
  return ok != 0;
}

// bounded wait: gives up after about WAIT_CYCLES SM cycles (32-bit clock, one
// wrap allowed) or when another role aborted, then raises the abort flag and
// records `code`.  Kept small in registers: the drain warps wait while holding
// their accumulator sums.
__device__ __forceinline__ bool mbar_wait(uint32_t a, uint32_t parity, volatile int* abort_flag, int* err,
                                          int code) {
  if (mbar_try(a, parity)) return true;
  const uint32_t t0 = static_cast<uint32_t>(clock());
  for (uint32_t spin = 1;; ++spin) {
    if (mbar_try_ns(a, parity, 1000u)) return true;
    if ((spin & 255u) == 0 &&
        (*abort_flag || static_cast<uint32_t>(clock()) - t0 > static_cast<uint32_t>(WAIT_CYCLES))) {
      if (!*abort_flag) {
        *abort_flag = 1;
        atomicExch(err, code);
      }
      return false;
    }
  }
}

// wait bounded by time alone (used on the way out, after an abort, for the
// kernel's own asynchronous copies and MMAs still in flight)
__device__ void mbar_wait_exit(uint32_t a, uint32_t parity, int* err) {
  const long long t0 = clock64();
  while (!mbar_try(a, parity)) {
    if (clock64() - t0 > WAIT_CYCLES) {
      atomicExch(err, 5);
      return;
    }
  }
}

// warp-level bounded wait: one lane polls the barrier, the other lanes wait at
// the __syncwarp (so that hundreds of threads do not spin on shared memory)
__device__ __forceinline__ bool mbar_wait_warp(uint32_t a, uint32_t parity, volatile int* abort_flag, int* err,
                                               int code) {
  int ok = 1;
  if ((threadIdx.x & 31) == 0) ok = mbar_wait(a, parity, abort_flag, err, code) ? 1 : 0;
  ok = __shfl_sync(0xffffffffu, ok, 0);
  return ok != 0;
}

__device__ __forceinline__ void mma(uint32_t d, uint64_t a, uint64_t b, uint32_t id, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d),
      "l"(a), "l"(b), "r"(id), "r"(acc)
      : "memory");
}

__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
               : "memory");
}

__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

}  // namespace
}  // namespace dmrg
