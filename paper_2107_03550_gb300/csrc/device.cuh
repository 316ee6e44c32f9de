// Small device helpers shared by the kernel translation units.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "kernels.cuh"

namespace sbiem {

// Programmatic dependent launch: a kernel launched with the programmatic
// serialization attribute may start while its predecessor runs; it must
// read nothing the predecessor chain writes before pdl_wait() returns.
// pdl_trigger() lets this kernel's own dependent start launching.  Both are
// no-ops for a kernel launched without the attribute.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Shared-memory address of a generic pointer into this CTA's shared memory.
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// Two FP32 fused multiply-adds in one packed instruction (fma.rn.f32x2):
// each lane rounds exactly as fmaf does.
__device__ __forceinline__ float2 ffma2(float2 a, float2 b, float2 c) {
  unsigned long long ra, rb, rc, rd;
  asm("mov.b64 %0, {%1, %2};" : "=l"(ra) : "f"(a.x), "f"(a.y));
  asm("mov.b64 %0, {%1, %2};" : "=l"(rb) : "f"(b.x), "f"(b.y));
  asm("mov.b64 %0, {%1, %2};" : "=l"(rc) : "f"(c.x), "f"(c.y));
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(rd) : "l"(ra), "l"(rb), "l"(rc));
  float2 d;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(d.x), "=f"(d.y) : "l"(rd));
  return d;
}

// Two FP32 additions in one packed instruction.
__device__ __forceinline__ float2 fadd2(float2 a, float2 b) {
  unsigned long long ra, rb, rd;
  asm("mov.b64 %0, {%1, %2};" : "=l"(ra) : "f"(a.x), "f"(a.y));
  asm("mov.b64 %0, {%1, %2};" : "=l"(rb) : "f"(b.x), "f"(b.y));
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(rd) : "l"(ra), "l"(rb));
  float2 d;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(d.x), "=f"(d.y) : "l"(rd));
  return d;
}

// s + c += a with the rounding error of the addition carried in c (Knuth's
// TwoSum; FP32 only -- an FP64 sum needs no compensation here).
__device__ __forceinline__ void two_sum_add(float& s, float& c, float a) {
  const float t = s + a;
  const float bb = t - s;
  c += (s - (t - bb)) + (a - bb);
  s = t;
}
__device__ __forceinline__ void two_sum_add(double& s, double& /*c*/, double a) { s += a; }

// Sum of four values over the warp with 9 additions instead of 20 (the FP64
// pipe is scarce): lanes exchange halves of the set first, so after two
// rounds a lane carries one value.  Lane 8 q returns value q; fixed order.
template <class T>
__device__ __forceinline__ T warp_reduce4(T v0, T v1, T v2, T v3) {
  const int lane = threadIdx.x & 31;
  const bool up = lane & 16, odd = lane & 8;
  const T a = (up ? v2 : v0) + __shfl_xor_sync(0xffffffffu, up ? v0 : v2, 16);
  const T b = (up ? v3 : v1) + __shfl_xor_sync(0xffffffffu, up ? v1 : v3, 16);
  T r = (odd ? b : a) + __shfl_xor_sync(0xffffffffu, odd ? a : b, 8);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
  return r;
}

// The bounded grid barrier of the persistent launches (every CTA resident):
// the last CTA to arrive resets the counter and advances the epoch, the
// others poll the epoch at most bar.limit times.  s_epoch (shared): the
// epoch read by thread 0 before any work.  False for a CTA that gave up: it
// has set SBIEM_FLAG_WAIT on every member and must leave.
template <class R>
__device__ __forceinline__ bool grid_barrier(const DevFault<R>* __restrict__ fs, const SweepBarrier& bar,
                                             const unsigned& s_epoch) {
  __shared__ unsigned s_fail;
  __syncthreads();
  if (threadIdx.x == 0) {
    s_fail = 0u;
    __threadfence();  // this CTA's partials before its arrival
    const unsigned ticket = atomicAdd(bar.count, 1u);
    if (ticket == gridDim.x - 1) {
      *reinterpret_cast<volatile unsigned*>(bar.count) = 0u;
      __threadfence();
      atomicAdd(bar.epoch, 1u);
    } else {
      bool released = false;
      for (long long q = 0; q < bar.limit; ++q) {
        if (*reinterpret_cast<volatile unsigned*>(bar.epoch) != s_epoch) {
          released = true;
          break;
        }
        __nanosleep(64);
      }
      if (!released) {
        s_fail = 1u;
        for (int r = 0; r < bar.members; ++r) atomicOr(fs[r].status, SBIEM_FLAG_WAIT);
      }
    }
    __threadfence();
  }
  __syncthreads();
  return s_fail == 0u;
}

}  // namespace sbiem
