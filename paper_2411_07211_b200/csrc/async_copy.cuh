// Asynchronous copies global -> shared memory and shared-memory barriers (inline PTX).
#pragma once

#include "common.cuh"

namespace b2 {

// Asynchronous 16-byte copy global -> shared memory of `bytes` (0 .. 16) bytes, the rest of the
// 16 zero-filled; element-sized copies for the vectors (bytes = 0: a zero).
__device__ __forceinline__ void cp_async16_full(void* dst, const void* src) {
  if (!B2_GUARD(src, 16)) {  // (bounds-checking build only: a zero-filled pack instead of the read)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, 0;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
    return;
  }
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async16(void* dst, const void* src, int bytes) {
  if (bytes > 0 && !B2_GUARD(src, (size_t)bytes)) bytes = 0;
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
               "r"(bytes)
               : "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_elem(void* dst, const void* src, bool valid) {
  if (valid && !B2_GUARD(src, (size_t)N)) valid = false;
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
               "n"(N), "r"(valid ? N : 0)
               : "memory");
}
// Shared-memory barriers (counting the bytes of bulk copies).
__device__ __forceinline__ void mbar_init(unsigned long long* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"((unsigned)__cvta_generic_to_shared(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect(unsigned long long* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"((unsigned)__cvta_generic_to_shared(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(unsigned long long* bar, unsigned parity) {
  unsigned done;
  asm volatile(
      "{\n\t.reg .pred q;\n\tmbarrier.try_wait.parity.shared::cta.b64 q, [%1], %2;\n\tselp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(done)
      : "r"((unsigned)__cvta_generic_to_shared(bar)), "r"(parity)
      : "memory");
  return done != 0;
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

}  // namespace b2
