// Double-float ("float-float") arithmetic: a value is an unevaluated sum hi + lo of two FP32 numbers with
// |lo| <= ulp(hi)/2, about 48 significant bits. Built from the error-free transformations
//   two_sum(a, b):  s = fl(a + b), e = (a - (s - bb)) + (b - bb), bb = s - a   (Knuth), a + b = s + e exactly;
//   two_prod(a, b): p = fl(a b),   e = fma(a, b, -p),                             a b = p + e exactly;
// (Dekker 1971; Hida, Li and Bailey, "Library for double-double and quad-double arithmetic", 2001).
// On GB300 the FP32 pipe is ~62x faster than the FP64 pipe, so the FP64-accurate block X of the mixed-precision solve is
// kept in this format, and its operator image is formed in it: ~10 FP32 operations per operation, a
// relative error of ~2^-44 instead of 2^-53, which the eigensolver does not resolve (its FP64 residual floor is
// ~1e-10 here).
#pragma once
#include <cuda_runtime.h>

namespace pc {

// packed FP32 pairs (add, mul, fma .f32x2: two results per instruction)
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 unpack2(f32x2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

struct df {
  float hi, lo;
};

__device__ __forceinline__ df df_from(double x) {
  df r;
  r.hi = (float)x;
  r.lo = (float)(x - (double)r.hi);
  return r;
}
__device__ __forceinline__ double df_to(df x) { return (double)x.hi + (double)x.lo; }

__device__ __forceinline__ df quick_two_sum(float a, float b) {  // requires |a| >= |b| (or a == 0)
  df r;
  r.hi = a + b;
  r.lo = b - (r.hi - a);
  return r;
}
__device__ __forceinline__ df two_sum(float a, float b) {
  df r;
  r.hi = a + b;
  const float bb = r.hi - a;
  r.lo = (a - (r.hi - bb)) + (b - bb);
  return r;
}
__device__ __forceinline__ df df_add(df x, df y) {
  const df s = two_sum(x.hi, y.hi);
  return quick_two_sum(s.hi, s.lo + (x.lo + y.lo));
}
__device__ __forceinline__ df df_neg(df x) { return df{-x.hi, -x.lo}; }
__device__ __forceinline__ df df_sub(df x, df y) { return df_add(x, df_neg(y)); }
__device__ __forceinline__ df df_mul(df x, df y) {
  const float p = x.hi * y.hi;
  float e = fmaf(x.hi, y.hi, -p);
  e = fmaf(x.hi, y.lo, e);
  e = fmaf(x.lo, y.hi, e);
  return quick_two_sum(p, e);
}

// complex double-float
struct cdf {
  df re, im;
};
__device__ __forceinline__ cdf cdf_from(double2 z) { return cdf{df_from(z.x), df_from(z.y)}; }
__device__ __forceinline__ double2 cdf_to(cdf z) { return make_double2(df_to(z.re), df_to(z.im)); }
__device__ __forceinline__ cdf cdf_add(cdf a, cdf b) { return cdf{df_add(a.re, b.re), df_add(a.im, b.im)}; }
__device__ __forceinline__ cdf cdf_sub(cdf a, cdf b) { return cdf{df_sub(a.re, b.re), df_sub(a.im, b.im)}; }
__device__ __forceinline__ cdf cdf_mul(cdf a, cdf b) {
  return cdf{df_sub(df_mul(a.re, b.re), df_mul(a.im, b.im)), df_add(df_mul(a.re, b.im), df_mul(a.im, b.re))};
}
// conj(a) * b
__device__ __forceinline__ cdf cdf_mulc(cdf a, cdf b) {
  return cdf{df_add(df_mul(a.re, b.re), df_mul(a.im, b.im)), df_sub(df_mul(a.re, b.im), df_mul(a.im, b.re))};
}
__device__ __forceinline__ cdf cdf_scale(cdf a, df s) { return cdf{df_mul(a.re, s), df_mul(a.im, s)}; }

// x + f for a double-float x and an FP32 f
__device__ __forceinline__ df df_addf(df x, float f) {
  const df s = two_sum(x.hi, f);
  return quick_two_sum(s.hi, s.lo + x.lo);
}

// Storage of complex double-float blocks. The solver keeps its FP64-accurate block as pairs (re.hi, re.lo, im.hi,
// im.lo) in one float4 (16 bytes, like complex128), so that its kernels read and write it without conversions:
// converting a double to a pair costs four FP64-pipe instructions and back three, more FP64 work than the
// double-float arithmetic does in FP32. complex128 blocks (the public entry points) convert on load and store.
__device__ __forceinline__ cdf ld_cdf(const double2 *p) { return cdf_from(*p); }
__device__ __forceinline__ cdf ld_cdf(const float4 *p) {
  const float4 v = *p;
  return cdf{df{v.x, v.y}, df{v.z, v.w}};
}
__device__ __forceinline__ void st_cdf(double2 *p, cdf z) { *p = cdf_to(z); }
__device__ __forceinline__ void st_cdf(float4 *p, cdf z) { *p = make_float4(z.re.hi, z.re.lo, z.im.hi, z.im.lo); }
// FP64 value of a stored element (for the FP64 checks and conversions off the iteration path)
__device__ __forceinline__ double2 ld_c128(const double2 *p) { return *p; }
__device__ __forceinline__ double2 ld_c128(const float2 *p) {
  const float2 v = *p;
  return make_double2((double)v.x, (double)v.y);
}
__device__ __forceinline__ double2 ld_c128(const float4 *p) {
  const float4 v = *p;
  return make_double2((double)v.x + (double)v.y, (double)v.z + (double)v.w);
}

}  // namespace pc
