// Double-float arithmetic: a value is the unevaluated sum hi + lo of two floats
// (about 48 significand bits), computed with FP32 instructions only.  GB300 runs
// FP64 at 1/64 of its FP32 rate, so the passes that need more than FP32 accuracy
// (right-hand side, refinement residual, outputs) can use this type instead.
//
// Error-free transformations (Knuth's two-sum, Dekker's fast two-sum, the FMA
// two-product) as in the double-double literature (Dekker 1971; Hida, Li & Bailey
// 2001).  Additions use the cheaper "sloppy" form: its error is bounded by about
// 2^-44 (|a| + |b|), which is what the pair sums need (an absolute error small
// compared with the summed magnitudes).
#pragma once

#include <cuda_runtime.h>

namespace gbi {

struct df {
  float hi, lo;
  df() = default;
  __host__ __device__ constexpr df(float h, float l) : hi(h), lo(l) {}
  // from a double constant (folded at compile time for literals)
  __host__ __device__ constexpr df(double d) : hi(float(d)), lo(float(d - double(float(d)))) {}
  __host__ __device__ constexpr df(int i) : hi(float(i)), lo(0.f) {}
  __host__ __device__ explicit operator float() const { return hi; }
};

// A product whose rounding error is formed separately (fmaf(a, b, -p)): it must stay rounded.  Left
// to itself the compiler may fuse it into a later sum -- s = p + e and e - (s - p) in df_fast_two_sum,
// p - (s - v) in df_two_sum -- which then holds the product's error a second time, so that the value
// is off by an FP32 rounding.  Whether it does depends on the code around it: the kernels as built were
// not hit, the same block in another kernel was (l <= 3 H/L off by 1e-8 of its norm).
__host__ __device__ __forceinline__ float df_rmul(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fmul_rn(a, b);
#else
  return a * b;
#endif
}

__host__ __device__ __forceinline__ df df_two_sum(float a, float b) {
  const float s = a + b;
  const float v = s - a;
  const float e = (a - (s - v)) + (b - v);
  return df(s, e);
}

__host__ __device__ __forceinline__ df df_fast_two_sum(float a, float b) {
  const float s = a + b;
  return df(s, b - (s - a));
}

__host__ __device__ __forceinline__ df df_two_prod(float a, float b) {
  const float p = df_rmul(a, b);
  return df(p, fmaf(a, b, -p));
}

// Sums and fused products leave the result unnormalised (lo is not folded back into
// hi): the exact two-sum of the high parts keeps hi + lo accurate, lo only collects
// rounding errors far below hi, and every consumer (products, sums, the conversion to
// double) uses hi and lo separately -- 3 FP32 operations fewer per operation.
__host__ __device__ __forceinline__ df operator+(df a, df b) {
  const df s = df_two_sum(a.hi, b.hi);
  return df(s.hi, s.lo + (a.lo + b.lo));
}

__host__ __device__ __forceinline__ df operator-(df a) { return df(-a.hi, -a.lo); }
__host__ __device__ __forceinline__ df operator-(df a, df b) { return a + (-b); }

__host__ __device__ __forceinline__ df operator*(df a, df b) {
  const float p = df_rmul(a.hi, b.hi);
  float e = fmaf(a.hi, b.hi, -p);
  e = fmaf(a.hi, b.lo, e);
  e = fmaf(a.lo, b.hi, e);
  return df_fast_two_sum(p, e);
}

__host__ __device__ __forceinline__ df& operator+=(df& a, df b) {
  a = a + b;
  return a;
}

// a * b + c in 10 FP32 operations.  With p = fl(a.hi b.hi), s = fl(p + c.hi) and Knuth's split
// v = s - p, w = s - v of the sum, both c.hi - v and p - w are exact and add up to p + c.hi - s; the
// product's error a.hi b.hi - p rides on the second one in a single FMA, a.hi b.hi - w.  (A product with
// its error followed by a two-sum takes 12.)  The double-float pair passes are bound by the FP32 pipe
// (70% busy), so operations are their time: with this, df_mul and df_rsqrt an H/H pair of l <= 3 takes
// 3650 instead of 4485 instructions, 151 us instead of 181 at N = 1024 (ncu); the error is at df_mul.
__host__ __device__ __forceinline__ df df_fma(df a, df b, df c) {
  const float p = df_rmul(a.hi, b.hi);
  const float s = p + c.hi;
  const float v = s - p;
  const float w = s - v;
  float e = (c.hi - v) + c.lo;
  e = fmaf(a.hi, b.lo, e);
  e = fmaf(a.lo, b.hi, e);
  return df(s, fmaf(a.hi, b.hi, -w) + e);
}

// a * b left unnormalised like the sums (4 operations, operator* 7): for a product that is added up
// at once -- the first one of a rotation's chains.  Factors use operator*, because the next product
// drops the two low parts' product, and so do the first products of the coupling sums.  Errors against
// FP64 as fractions of those with every product normalised and 12 operations per fused product (which
// this replaced), over 10^5 pairs in each of 108 sets: l <= 2, 3, 4; H/H, H/L, L/all; 2-6, 6-60, 60-300 and
// 300-3000 radii apart; all directions, near the xy plane, near the z axis.  The block itself: median 0.83-1.01,
// rms 0.63-0.82, 99th percentile 0.54-0.72, largest 0.43-0.80.  Its product with random coefficients: rms
// 0.67-0.96, 99th percentile 0.61-0.89, largest 0.35-0.92, median 0.89-1.05 for H/H and H/L and up to 1.12 for
// L/all.  (Factors and coupling sums unnormalised too: medians of H/H up to 1.22.)
__host__ __device__ __forceinline__ df df_mul(df a, df b) {
  const float p = df_rmul(a.hi, b.hi);
  float e = fmaf(a.hi, b.hi, -p);
  e = fmaf(a.hi, b.lo, e);
  e = fmaf(a.lo, b.hi, e);
  return df(p, e);
}

// with a factor that is exact in FP32: no a.lo b.hi term
__host__ __device__ __forceinline__ df df_fma(float a, df b, df c) {
  const float p = df_rmul(a, b.hi);
  const float s = p + c.hi;
  const float v = s - p;
  const float w = s - v;
  const float e = fmaf(a, b.lo, (c.hi - v) + c.lo);
  return df(s, fmaf(a, b.hi, -w) + e);
}
__host__ __device__ __forceinline__ df df_mul(float a, df b) {
  const float p = df_rmul(a, b.hi);
  return df(p, fmaf(a, b.lo, fmaf(a, b.hi, -p)));
}

__host__ __device__ __forceinline__ bool operator>(df a, df b) {
  return a.hi > b.hi || (a.hi == b.hi && a.lo > b.lo);
}

__host__ __device__ __forceinline__ double df_to_double(df a) { return double(a.hi) + double(a.lo); }

// 1/sqrt(a): FP32 estimate y, residual r = 1 - a y^2 (one FMA each for the parts of a and y^2), then
// y (1 + r/2 + 3 r^2/8).  r is some 2^-22, so FP32 carries the correction (11 operations; a Newton step in
// double-float took 33 and left the r^2 term out).
__host__ __device__ __forceinline__ df df_rsqrt(df a) {
#ifdef __CUDA_ARCH__
  const float y = rsqrtf(a.hi);
#else
  const float y = 1.0f / sqrtf(a.hi);
#endif
  const float q = df_rmul(y, y);
  const float ql = fmaf(y, y, -q);
  float r = fmaf(-a.hi, q, 1.0f);
  r = fmaf(-a.hi, ql, r);
  r = fmaf(-a.lo, q, r);
  return df_fast_two_sum(y, y * (r * fmaf(0.375f, r, 0.5f)));
}

#ifdef __CUDACC__
__device__ __forceinline__ df df_shfl_xor(df v, int o) {
  return df(__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o));
}
#endif

}  // namespace gbi

// a * b + c in the arithmetic of T (fused where the type has a fused form); the
// generated pair-frame code chains its sums of products through this.  A float first factor is a
// constant that is exact in FP32.
__host__ __device__ __forceinline__ float gbi_fmac(float a, float b, float c) { return fmaf(a, b, c); }
__host__ __device__ __forceinline__ double gbi_fmac(double a, double b, double c) { return fma(a, b, c); }
__host__ __device__ __forceinline__ double gbi_fmac(float a, double b, double c) { return fma(double(a), b, c); }
__host__ __device__ __forceinline__ gbi::df gbi_fmac(gbi::df a, gbi::df b, gbi::df c) { return gbi::df_fma(a, b, c); }
__host__ __device__ __forceinline__ gbi::df gbi_fmac(float a, gbi::df b, gbi::df c) { return gbi::df_fma(a, b, c); }
// a * b that is added up or used as a factor once or twice
__host__ __device__ __forceinline__ float gbi_mul(float a, float b) { return a * b; }
__host__ __device__ __forceinline__ double gbi_mul(double a, double b) { return a * b; }
__host__ __device__ __forceinline__ double gbi_mul(float a, double b) { return double(a) * b; }
__host__ __device__ __forceinline__ gbi::df gbi_mul(gbi::df a, gbi::df b) { return gbi::df_mul(a, b); }
__host__ __device__ __forceinline__ gbi::df gbi_mul(float a, gbi::df b) { return gbi::df_mul(a, b); }
