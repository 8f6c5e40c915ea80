// Two FP32 values per instruction (the paired FFMA2 / FMUL2 / FADD2 of sm_100 and later).
// Each element is rounded exactly as the scalar operation rounds it, so a paired pass gives the
// scalar pass's results bit for bit; it halves the issued FP32 instructions, not the FMA pipe's
// work (a paired FMA occupies the pipe for two lanes' worth).
#pragma once

#include <cuda_runtime.h>

namespace gbi {

struct f2 {
  float2 v;
  __device__ __forceinline__ f2() {}
  __device__ __forceinline__ explicit f2(float s) : v(make_float2(s, s)) {}
  __device__ __forceinline__ f2(float a, float b) : v(make_float2(a, b)) {}
  __device__ __forceinline__ explicit f2(float2 p) : v(p) {}
};
__device__ __forceinline__ f2 operator+(f2 a, f2 b) { return f2(__fadd2_rn(a.v, b.v)); }
__device__ __forceinline__ f2 operator*(f2 a, f2 b) { return f2(__fmul2_rn(a.v, b.v)); }
__device__ __forceinline__ f2 operator-(f2 a) { return f2(-a.v.x, -a.v.y); }
__device__ __forceinline__ f2 operator-(f2 a, f2 b) { return a + (-b); }
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) { return f2(__ffma2_rn(a.v, b.v, c.v)); }
__device__ __forceinline__ f2 rsqrt2(f2 a) { return f2(rsqrtf(a.v.x), rsqrtf(a.v.y)); }
// the scalar counterparts, for code written once for both
__device__ __forceinline__ float fma2(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ float rsqrt2(float a) { return rsqrtf(a); }

}  // namespace gbi
