// Pushes between the CTAs of a cluster (sm_103a): stores into another CTA's
// shared memory that complete on that CTA's mbarrier, and the bounded wait
// for them.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

namespace bbp {
namespace {

__device__ __forceinline__ uint32_t saddr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t remote(uint32_t a, int rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}

// Pushes of eight or sixteen bytes into another CTA's shared memory that
// complete on that CTA's mbarrier, and the bounded wait for them: a wait that
// runs out marks the CTA (the kernels report it: NaN in the panels, the status
// word in the Jacobi).
__device__ __forceinline__ void push(uint32_t a, uint32_t bar, float v0, float v1) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];" ::"r"(a),
               "f"(v0), "f"(v1), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void push(uint32_t a, uint32_t bar, float v0, float v1, float v2, float v3) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(a),
               "f"(v0), "f"(v1), "f"(v2), "f"(v3), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void push(uint32_t a, uint32_t bar, double v0, double v1) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.f64 [%0], {%1, %2}, [%3];" ::"r"(a),
               "d"(v0), "d"(v1), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void bar_init(uint32_t bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void bar_expect(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool bar_try(uint32_t bar, uint32_t phase) {
  uint32_t ok;
  asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
               : "=r"(ok)
               : "r"(bar), "r"(phase)
               : "memory");
  return ok != 0;
}
__device__ __forceinline__ void bar_wait(uint32_t bar, uint32_t phase, volatile int* failed) {
  if (bar_try(bar, phase)) return;
  unsigned long long t0, t1;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
  while (!bar_try(bar, phase)) {
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t1));
    if (*failed || t1 - t0 > 2000000000ull) {
      *failed = 1;
      return;
    }
  }
}

__device__ __forceinline__ void push128(uint32_t a, uint32_t bar, float4 v) { push(a, bar, v.x, v.y, v.z, v.w); }
__device__ __forceinline__ float4 lds128(uint32_t a) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a));
  return v;
}
__device__ __forceinline__ void sts128(uint32_t a, float4 v) {
  asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}

}  // namespace
}  // namespace bbp
