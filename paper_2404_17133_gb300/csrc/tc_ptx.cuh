// Inline-PTX helpers shared by the tcgen05 kernels: mbarriers with bounded
// waits, the K-major 128-byte-swizzle shared-memory descriptor and the MMA
// completion commit.
#pragma once
#include <cstdint>

namespace tddft {
namespace {

// A wait on an mbarrier gives up after WAIT_NS (the kernel then records an error
// code and leaves its loop; the host reports TDDFT_ERR_CUDA).  The limit is a time:
// a number of polls is none, since a poll may suspend its thread for as long as the
// hardware chooses.  POLL_NS bounds one suspension; the clock is read only
// after a poll that found the phase open.  The longest wait of a kernel that works
// is for its CTA's whole K range, some milliseconds.
constexpr unsigned long long WAIT_NS = 2000000000ull;
constexpr uint32_t POLL_NS = 1000000u;

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}

__device__ __forceinline__ bool mbar_poll(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity), "r"(POLL_NS)
      : "memory");
  return ok != 0;
}

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Bounded wait for the completion of phase `parity`; false on timeout.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
  const uint32_t a = smem_u32(bar);
  if (mbar_poll(a, parity)) return true;
  const unsigned long long t0 = global_ns();
  do {
    if (mbar_poll(a, parity)) return true;
  } while (global_ns() - t0 < WAIT_NS);
  return false;
}

// Shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row groups 1024 B apart.
__device__ __forceinline__ uint64_t sdesc(const void* p) {
  const uint64_t addr = smem_u32(p);
  return ((addr & 0x3FFFFull) >> 4) | (1ull << 16) | ((uint64_t)(1024 >> 4) << 32) | (1ull << 46) |
         (2ull << 61);
}

// Arrive on `bar` when every tcgen05.mma this thread issued so far has completed.
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                   smem_u32(bar))
               : "memory");
}

}  // namespace
}  // namespace tddft
