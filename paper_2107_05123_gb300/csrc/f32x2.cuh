// Pairs of FP32 numbers in one 64-bit register pair. The packed instructions of sm_10x (FADD2,
// FMUL2, FFMA2) do two FP32 operations, each rounded as the scalar one, in one issue slot; the
// FP32 applies are bound by instruction issue, so their element arithmetic runs on two elements
// at a time.
#pragma once

#include <cuda_runtime.h>

namespace chns {

struct __align__(8) F2 {
  float x, y;
  F2() = default;
  __host__ __device__ F2(float a) : x(a), y(a) {}
  __host__ __device__ F2(float a, float b) : x(a), y(b) {}
};

__device__ __forceinline__ float2 raw(F2 a) { return make_float2(a.x, a.y); }
__device__ __forceinline__ F2 from_raw(float2 a) { return F2(a.x, a.y); }

__device__ __forceinline__ F2 mad(F2 a, F2 b, F2 c) {
  return from_raw(__ffma2_rn(raw(a), raw(b), raw(c)));
}
__device__ __forceinline__ F2 operator+(F2 a, F2 b) { return from_raw(__fadd2_rn(raw(a), raw(b))); }
__device__ __forceinline__ F2 operator*(F2 a, F2 b) { return from_raw(__fmul2_rn(raw(a), raw(b))); }
__device__ __forceinline__ F2 operator-(F2 a) { return F2(-a.x, -a.y); }
__device__ __forceinline__ F2 operator-(F2 a, F2 b) { return a + (-b); }
__device__ __forceinline__ F2& operator+=(F2& a, F2 b) { return a = a + b; }
__device__ __forceinline__ F2& operator-=(F2& a, F2 b) { return a = a - b; }
__device__ __forceinline__ F2& operator*=(F2& a, F2 b) { return a = a * b; }

// min(max(v, lo), hi) that keeps NaN
__device__ __forceinline__ float clamp_nan(float v, float lo, float hi) {
  float r;
  asm("{\n\t.reg .f32 t;\n\tmax.NaN.f32 t, %1, %2;\n\tmin.NaN.f32 %0, t, %3;\n\t}"
      : "=f"(r)
      : "f"(v), "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ F2 clamp_nan(F2 v, float lo, float hi) {
  return F2(clamp_nan(v.x, lo, hi), clamp_nan(v.y, lo, hi));
}

// 1/v to one ulp (the hardware approximation; FP32 applies feed FP64-refined solves)
__device__ __forceinline__ float rcp_approx(float v) {
  float r;
  asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(v));
  return r;
}
__device__ __forceinline__ F2 rcp_approx(F2 v) { return F2(rcp_approx(v.x), rcp_approx(v.y)); }

}  // namespace chns
