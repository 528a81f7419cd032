// Two FP32 values in one 64-bit register pair, the operand of Blackwell's packed FP32 instructions
// (add / mul / fma .f32x2). One instruction works on both; the FMA rate is that of scalar FP32 (both
// measured at 3.4-3.5 scalar FMAs per clock and SM sub-partition group on GB300), so what a packed
// kernel saves is half of the issue slots, which bound the collision. Every operation rounds each
// half exactly as its scalar counterpart.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <cstring>

namespace lbm {

struct alignas(8) F2 {
  uint64_t v;
  F2() = default;
  __host__ __device__ __forceinline__ F2(float a, float b) {
#ifdef __CUDA_ARCH__
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(a), "f"(b));
#else
    uint32_t lo, hi;
    std::memcpy(&lo, &a, 4);
    std::memcpy(&hi, &b, 4);
    v = uint64_t(lo) | (uint64_t(hi) << 32);
#endif
  }
  __host__ __device__ __forceinline__ explicit F2(float s) : F2(s, s) {}
  __host__ __device__ __forceinline__ explicit F2(double s) : F2(float(s)) {}
  __host__ __device__ __forceinline__ explicit F2(int s) : F2(float(s)) {}
  __device__ __forceinline__ void get(float& a, float& b) const { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
};
__device__ __forceinline__ F2 operator+(F2 a, F2 b) {
  F2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 operator-(F2 a, F2 b) {
  F2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) {
  F2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
__device__ __forceinline__ F2 operator*(F2 a, F2 b) {
  F2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 operator/(F2 a, F2 b) {
  float a0, a1, b0, b1;
  a.get(a0, a1);
  b.get(b0, b1);
  return F2(a0 / b0, a1 / b1);
}

}  // namespace lbm
