// tcgen05 (tensor cores with accumulators in TMEM), mbarriers and fixed-point operands: what the
// tensor-core kernels share (gram_tc.cu, update_tc.cu).
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>

namespace pbs {

constexpr unsigned kSpinLimit = 1u << 20;  // tries (of 2 us at most) after which a wait gives up
constexpr int kExpInf = 100000;            // exponent of a column with a non-finite value
constexpr int kMinExp = -900;              // columns below 2^kMinExp count as zero

__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(unsigned bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try(unsigned bar, unsigned parity) {  // suspends the thread for a while
  unsigned ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cta.shared::cta.b64 p, [%1], %2, %3;\n\tselp.u32 %0, 1, "
      "0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity), "r"(2000u)
      : "memory");
  return ok != 0;
}
// Waits for the phase of the given parity; gives up after kSpinLimit tries and sets *abort, after
// which no wait of the CTA blocks any more (the result is then marked invalid).
__device__ __forceinline__ void mbar_wait(unsigned bar, unsigned parity, volatile int* abort) {
  for (unsigned t = 0; !mbar_try(bar, parity); ++t) {
    if (*abort) return;
    if (t == kSpinLimit) {
      *abort = 1;
      return;
    }
  }
}
__device__ __forceinline__ void tc_mma(unsigned d, unsigned long long a, unsigned long long b, unsigned idesc,
                                       unsigned accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void tc_commit(unsigned bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_ld16(unsigned addr, float (&v)[16]) {
  unsigned r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, "
      "[%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(addr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int k = 0; k < 16; ++k) v[k] = __uint_as_float(r[k]);
}
__device__ __forceinline__ void tc_ld4(unsigned addr, float (&v)[4]) {
  unsigned r[4];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int k = 0; k < 4; ++k) v[k] = __uint_as_float(r[k]);
}
__device__ __forceinline__ void tc_ld8(unsigned addr, float (&v)[8]) {
  unsigned r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(addr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int k = 0; k < 8; ++k) v[k] = __uint_as_float(r[k]);
}
// Shared-memory descriptor: K-major, no swizzle; rows in groups of 8 (128 bytes each, consecutive),
// columns of 8 binary16 values `octet` bytes apart.
__device__ __forceinline__ unsigned long long tc_desc(unsigned addr, unsigned octet) {
  return (unsigned long long)((addr >> 4) & 0x3FFFu) | ((unsigned long long)(octet >> 4) << 16) |
         ((unsigned long long)(128 >> 4) << 32) | (1ull << 46);
}
// Instruction descriptor: binary16 operands, FP32 sums, M = 128, N = n.
__host__ __device__ __forceinline__ constexpr unsigned tc_idesc(unsigned n) { return (1u << 4) | ((n >> 3) << 17) | (8u << 24); }

}  // namespace pbs
