// ptx.cuh -- inline PTX for the staged kernels: 16-byte cp.async copies from global to shared
// memory, completion tracked per thread in commit groups (nothing waits on another thread).
#pragma once

#ifndef __CUDACC_RTC__
#include <cstdint>
#endif

namespace adha {

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// 16-byte asynchronous copy global -> shared (LDGSTS), completion tracked per thread in groups.
__device__ __forceinline__ void cp_async16(void* sdst, const void* gsrc) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(sdst)), "l"(gsrc) : "memory");
}

// The same with the shared address already formed.
__device__ __forceinline__ void cp_async16_at(uint32_t sdst, const void* gsrc) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sdst), "l"(gsrc) : "memory");
}

// A 16-byte copy of which only the first `bytes` are read (the rest of the destination is zeroed).
__device__ __forceinline__ void cp_async16_part(uint32_t sdst, const void* gsrc, int bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(sdst), "l"(gsrc), "r"(bytes) : "memory");
}

__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }

// Wait until at most N of this thread's committed cp.async groups are pending.
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Two fp32 values in one 64-bit register (low half first).  The packed instructions (sm_100 and
// later) compute both halves in one issue slot, each an IEEE fp32 operation rounded to nearest
// on its own (no flush to zero), so a pair gives the bits of the two scalar operations.  There is no
// packed product here: see f2_mul_alone.
__device__ __forceinline__ unsigned long long f2_pack(float lo, float hi) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void f2_unpack(unsigned long long v, float* lo, float* hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(*lo), "=f"(*hi) : "l"(v));
}
__device__ __forceinline__ unsigned long long f2_sub_rn(unsigned long long a, unsigned long long b) {
  unsigned long long r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ unsigned long long f2_fma_rn(unsigned long long a, unsigned long long b, unsigned long long c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ unsigned long long f2_add_rn(unsigned long long a, unsigned long long b) {
  unsigned long long r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

// 1/x within an ulp.
__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// a * b rounded on its own, as fma(a, b, -0): ptxas contracts mul.rn.f32x2 followed by add.rn.f32x2 (or
// sub) into one fma, whatever -fmad says (measured: equal to fmaf on 4096 of 4096 random pairs,
// to the separate operations on 3229), so a product that is added to must not be a mul.  neg_zero
// is the pair (-0, -0), passed through the kernel's arguments: as a literal it could be folded away.
__device__ __forceinline__ unsigned long long f2_mul_alone(unsigned long long a, unsigned long long b,
                                                           unsigned long long neg_zero) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(neg_zero));
  return r;
}

}  // namespace adha
