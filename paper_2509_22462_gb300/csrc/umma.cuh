// tcgen05 / TMEM primitives of the tensor-core kernels (inline PTX for sm_103a), beside async.cuh.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <cstdint>

#include "async.cuh"

namespace nnc {
namespace umma {

using async::griddep_launch;
using async::griddep_wait;
using async::kWaitCycles;
using async::mbar_arrive;
using async::mbar_expect_tx;
using async::mbar_init;
using async::mbar_try;
using async::smem_u32;
using async::tma_load_2d;

// Bounded wait for the phase with the given parity.  Returns false if the CTA aborted or the
// wait ran out (then the error word, which there always is here, and the CTA's abort flag are set).  Going
// through async::mbar_wait_abort costs 0.6 % of 784 -> 4096 x 7 -> 10 in the FP64 form.
__device__ __forceinline__ bool mbar_wait(uint32_t a, uint32_t parity, int* err, int code,
                                          volatile int* abort_flag, long long limit = kWaitCycles) {
  if (mbar_try(a, parity)) return true;
  const long long t0 = clock64();
  while (true) {
    if (mbar_try(a, parity)) return true;
    if (*abort_flag) return false;
    if (clock64() - t0 > limit) {
      atomicCAS(err, 0, code);
      *abort_flag = 1;
      return false;
    }
  }
}

// Shared-memory matrix descriptor of tcgen05 for a K-major tile written by TMA with 128- or
// 64-byte swizzling: start address >> 4 (bits 0-13), stride between 8-row groups (SBO, >> 4 at
// bit 32), descriptor version 1 (bit 46), layout SWIZZLE_128B (2) or SWIZZLE_64B (4) at bits
// 61-63.  Moving along K inside a swizzled row is done by advancing the start address (32 bytes
// per K = 16).
template <int SWZ, int SBO>
__device__ __forceinline__ uint64_t sdesc(uint32_t addr) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)(SBO >> 4) << 32) | (1ull << 46) |
         ((uint64_t)SWZ << 61);
}

__device__ __forceinline__ void umma_bf16(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t idesc,
                                          uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem_d),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ void umma_f8(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t idesc,
                                        uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem_d),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ void umma_commit(uint32_t mbar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar)
      : "memory");
}

__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// True on every thread of the four epilogue warps (named barrier 1, 128 threads) only if p is
// true on all of them, so that the barriers of the staged epilogue are reached by all or none.
__device__ __forceinline__ bool epi_all(bool p) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred q;\n\t"
      "setp.ne.u32 q, %1, 0;\n\t"
      "bar.red.and.pred q, 1, 128, q;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}\n"
      : "=r"(r)
      : "r"((uint32_t)p)
      : "memory");
  return r != 0;
}

__device__ __forceinline__ void epi_sync() { asm volatile("bar.sync 1, 128;" ::: "memory"); }

}  // namespace umma
}  // namespace nnc
