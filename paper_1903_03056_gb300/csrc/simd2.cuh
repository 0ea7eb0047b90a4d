// Pairs of FP32 values in one 64-bit register pair: Blackwell adds, multiplies and multiply-adds
// both halves with one instruction (each half rounded as the scalar instruction rounds it).
#pragma once

#include <cuda_runtime.h>

#include "fft_line.cuh"

namespace dgfs {

struct F2 {
  unsigned long long v;
};

__device__ __forceinline__ F2 pack2(float lo, float hi) {
  F2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float2 unpack2(F2 a) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a.v));
  return r;
}
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
__device__ __forceinline__ F2 operator*(F2 a, F2 b) {
  F2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) {
  F2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
__device__ __forceinline__ F2 operator-(F2 a) { return a * pack2(-1.0f, -1.0f); }

// complex values with packed parts: two independent complex numbers per element
struct C2 {
  F2 x, y;
};
template <> struct cplx_t<F2> { using type = C2; };
template <> struct real_const<F2> { using type = float; };

__device__ __forceinline__ F2 mulc(F2 a, float c) { return a * pack2(c, c); }
__device__ __forceinline__ F2 fmac(F2 a, float c, F2 b) { return fma2(a, pack2(c, c), b); }

}  // namespace dgfs
