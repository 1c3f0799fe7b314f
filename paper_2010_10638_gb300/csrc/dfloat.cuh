// Double-float accumulation of exact FP32 products, shared by the QRP kernels.
//
// s += a * (bh + bl), where bh + bl is an FP64 value split into two floats.  a * bh is
// formed exactly as p + e (FMA residual), p is added to the running high part with
// TwoSum (Knuth), and every rounding error goes into the low part.  With a flush of
// (hi + lo) into an FP64 sum every few hundred terms the relative error of a dot
// product stays near 2^-46, while every operation runs on the FP32 pipe.
#pragma once

namespace tk {

struct DF {
  float hi = 0.f, lo = 0.f;
};

__device__ __forceinline__ void df_fma(DF &s, float a, float bh, float bl) {
  const float p = a * bh;
  const float e = fmaf(a, bh, -p);
  const float q = a * bl;
  const float t = s.hi + p;
  const float bp = t - s.hi;
  const float err = (s.hi - (t - bp)) + (p - bp);
  s.hi = t;
  s.lo += err + (e + q);
}

// double-float addition a += b (TwoSum of the high parts, then renormalisation)
__device__ __forceinline__ void df_add(DF &a, const DF b) {
  const float s = a.hi + b.hi;
  const float bp = s - a.hi;
  float e = (a.hi - (s - bp)) + (b.hi - bp);
  e += a.lo + b.lo;
  a.hi = s + e;
  a.lo = e - (a.hi - s);
}

// an FP64 value as a pair
__device__ __forceinline__ float2 df2_of(double v) {
  const float h = __double2float_rn(v);
  return make_float2(h, __double2float_rn(v - (double)h));
}
// t -= (v.x + v.y) (m.x + m.y): the product of the high parts exactly (FMA residual), the
// cross terms by FMA, the low-low term dropped (2^-48 of the product); TwoSum of the high parts
__device__ __forceinline__ void df_sub_prod(DF &t, float2 v, float2 m) {
  const float p = v.x * m.x;
  float e = fmaf(v.x, m.x, -p);
  e = fmaf(v.x, m.y, e);
  e = fmaf(v.y, m.x, e);
  const float s = t.hi - p;
  const float bp = s - t.hi;
  const float err = (t.hi - (s - bp)) - (p + bp);
  t.hi = s;
  t.lo += err - e;
}

// FP32 -> FP64 without the FP64 pipe: the same sign, the exponent rebiased (+896), the
// mantissa shifted up 29 bits; exact for normal numbers (zero, subnormals, inf and NaN
// take the conversion instruction)
__device__ __forceinline__ double f2d_exact(float f) {
  const unsigned b = __float_as_uint(f);
  const unsigned e = (b >> 23) & 0xffu;
  if (e == 0u || e == 0xffu) return (double)f;
  const unsigned long long d = ((unsigned long long)(b & 0x80000000u) << 32) |
                               ((unsigned long long)(e + 896u) << 52) | ((unsigned long long)(b & 0x7fffffu) << 29);
  return __longlong_as_double((long long)d);
}

}  // namespace tk
