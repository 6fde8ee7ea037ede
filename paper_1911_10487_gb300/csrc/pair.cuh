// Two independent FP32 values in one 64-bit register pair, and the packed arithmetic on them
// (add, sub, mul, fma .rn.f32x2: each half rounded as the scalar operation).  A packed instruction
// does two operations for one issue slot at the FP32 pipe's unchanged rate, so it helps a kernel whose
// schedulers are busy with loads, addresses and shared memory beside the arithmetic.
#pragma once
#include "common.cuh"

namespace fl {

struct __align__(8) f2 {
  unsigned long long v;
  f2() = default;
  __device__ __forceinline__ explicit f2(unsigned long long b) : v(b) {}
  __device__ __forceinline__ f2(float a, float b) { asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(a), "f"(b)); }
  __device__ __forceinline__ explicit f2(float a) : f2(a, a) {}
  __device__ __forceinline__ explicit f2(double a) : f2((float)a, (float)a) {}
  __device__ __forceinline__ explicit f2(int a) : f2((float)a, (float)a) {}
  __device__ __forceinline__ float2 split() const {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
  }
  __device__ __forceinline__ friend f2 fma(f2 a, f2 b, f2 c) {
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
  }
};
__device__ __forceinline__ f2 operator+(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 operator-(f2 a, f2 b) {
  f2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 operator*(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 operator-(f2 a) { return f2(a.v ^ 0x8000000080000000ull); }

// two complex values: their real parts and their imaginary parts
struct __align__(16) cf2 {
  f2 x, y;
};
template <> struct cx_t<f2> { using type = cf2; };
__device__ __forceinline__ cf2 pair_of(float2 a, float2 b) { return cf2{f2(a.x, b.x), f2(a.y, b.y)}; }
__device__ __forceinline__ cf2 operator+(cf2 a, cf2 b) { return cf2{a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ cf2 operator-(cf2 a, cf2 b) { return cf2{a.x - b.x, a.y - b.y}; }
__device__ __forceinline__ cf2 operator*(cf2 a, cf2 w) {
  return cf2{a.x * w.x - a.y * w.y, fma(a.x, w.y, a.y * w.x)};
}
template <bool INV> __device__ __forceinline__ cf2 rot90(cf2 a) {
  return INV ? cf2{-a.y, a.x} : cf2{a.y, -a.x};
}

}  // namespace fl
