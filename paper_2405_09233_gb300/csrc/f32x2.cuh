// Two FP32 values in one 64-bit register, and the instructions that work on both at once.
#pragma once
#include <cmath>
#include <cstring>
#include <cuda_runtime.h>

namespace ts {

using f32x2 = unsigned long long;   // two packed FP32 values
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f32x2 dup2(float v) {
  f32x2 d;
  asm("mov.b64 %0, {%1, %1};" : "=l"(d) : "f"(v));
  return d;
}
__device__ __forceinline__ void split2(f32x2 v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}

// The same as a number type: code written for float runs on it two values at a time (on the host value by value).
struct F2 {
  f32x2 v = 0ull;
};
__host__ __device__ __forceinline__ F2 make_f2(float lo, float hi) {
  F2 r;
#ifdef __CUDA_ARCH__
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
#else
  float q[2] = {lo, hi};
  memcpy(&r.v, q, sizeof(q));
#endif
  return r;
}
__host__ __device__ __forceinline__ void split(F2 a, float& lo, float& hi) {
#ifdef __CUDA_ARCH__
  split2(a.v, lo, hi);
#else
  float q[2];
  memcpy(q, &a.v, sizeof(q));
  lo = q[0];
  hi = q[1];
#endif
}
__host__ __device__ __forceinline__ F2 fma_t(F2 a, F2 b, F2 c) {
#ifdef __CUDA_ARCH__
  return F2{fma2(a.v, b.v, c.v)};
#else
  float x[2], y[2], z[2];
  split(a, x[0], x[1]);
  split(b, y[0], y[1]);
  split(c, z[0], z[1]);
  return make_f2(fmaf(x[0], y[0], z[0]), fmaf(x[1], y[1], z[1]));
#endif
}
__host__ __device__ __forceinline__ F2 operator+(F2 a, F2 b) {
#ifdef __CUDA_ARCH__
  return F2{add2(a.v, b.v)};
#else
  float x[2], y[2];
  split(a, x[0], x[1]);
  split(b, y[0], y[1]);
  return make_f2(x[0] + y[0], x[1] + y[1]);
#endif
}
__host__ __device__ __forceinline__ F2 operator*(F2 a, F2 b) {
#ifdef __CUDA_ARCH__
  F2 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d.v) : "l"(a.v), "l"(b.v));
  return d;
#else
  float x[2], y[2];
  split(a, x[0], x[1]);
  split(b, y[0], y[1]);
  return make_f2(x[0] * y[0], x[1] * y[1]);
#endif
}
__host__ __device__ __forceinline__ F2 operator-(F2 a, F2 b) { return fma_t(b, make_f2(-1.f, -1.f), a); }

}  // namespace ts
