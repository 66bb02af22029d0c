// df32.cuh -- double-float ("float-float") arithmetic for kernels whose FP64 work would
// run on GB300's FP64 pipe (1/64 of the FP32 rate).  A value is the unevaluated sum
// hi + lo of two floats with |lo| <= ulp(hi) / 2: about 48 significant bits, exponent range
// of float.  Built on the classical error-free transformations:
//   TwoSum (Knuth, TAOCP vol. 2, 4.2.2): s + e = a + b exactly, any a, b;
//   Fast2Sum (Dekker 1971): the same when |a| >= |b|, three operations;
//   TwoProduct with a fused multiply-add: p + e = a b exactly, e = fma(a, b, -p).
// The sum carries the low parts' rounding error too (accurate under cancellation, which
// the finite-element differences u_b - u_(1-b) and the element sums produce); the product
// drops lo * lo.  Relative error of one operation: a few 2^-48.
#pragma once

#include <cstdint>

#include <cuda_runtime.h>

struct df {
  float hi, lo;
  df() = default;
  __host__ __device__ constexpr df(float h, float l) : hi(h), lo(l) {}
  __host__ __device__ explicit constexpr df(int x) : hi((float)x), lo(0.0f) {}
  // rounded split of a double (exact for constants folded at compile time)
  __host__ __device__ explicit df(double x) : hi((float)x), lo((float)(x - (double)(float)x)) {}
};

__host__ __device__ __forceinline__ df df_two_sum(float a, float b) {
  const float s = a + b;
  const float bb = s - a;
  return df(s, (a - (s - bb)) + (b - bb));
}
__host__ __device__ __forceinline__ df df_fast_two_sum(float a, float b) {
  const float s = a + b;
  return df(s, b - (s - a));
}
__host__ __device__ __forceinline__ df df_two_prod(float a, float b) {
  const float p = a * b;
  return df(p, fmaf(a, b, -p));
}

__host__ __device__ __forceinline__ df operator+(df a, df b) {
  df s = df_two_sum(a.hi, b.hi);
  const df t = df_two_sum(a.lo, b.lo);
  s = df_fast_two_sum(s.hi, s.lo + t.hi);
  return df_fast_two_sum(s.hi, s.lo + t.lo);
}
__host__ __device__ __forceinline__ df operator-(df a) { return df(-a.hi, -a.lo); }
__host__ __device__ __forceinline__ df operator-(df a, df b) { return a + (-b); }
__host__ __device__ __forceinline__ df operator*(df a, df b) {
  const df p = df_two_prod(a.hi, b.hi);
  return df_fast_two_sum(p.hi, fmaf(a.hi, b.lo, fmaf(a.lo, b.hi, p.lo)));
}
__host__ __device__ __forceinline__ df& operator+=(df& a, df b) { return a = a + b; }
__host__ __device__ __forceinline__ df fma(df a, df b, df c) { return a * b + c; }

// 1 / sqrt(x), x > 0: the float estimate y refined by one step of third order,
// y (1 + e / 2 + 3 e^2 / 8) with e = 1 - x y^2 (about 2^-22; 1 - hi is exact there); the
// neglected term is 5 e^3 / 16, below 2^-66
__device__ __forceinline__ df inv_sqrt(df x) {
  const float y = rsqrtf(x.hi);
  const df p = x * df_two_prod(y, y);
  const df e = df_two_sum(1.0f - p.hi, -p.lo);
  const float yh = 0.5f * y;
  const df c = df_two_prod(yh, e.hi);
  const df s = df_fast_two_sum(y, c.hi);
  return df_fast_two_sum(s.hi, s.lo + fmaf(yh, e.lo, fmaf(0.75f * yh * e.hi, e.hi, c.lo)));
}
__device__ __forceinline__ float inv_sqrt(float x) { return rsqrtf(x); }
__device__ __forceinline__ double inv_sqrt(double x) { return rsqrt(x); }

// Quick sum and fused multiply-add: the low parts are summed in one float, so the error is
// a few 2^-48 of the operands instead of the result (11 operations against 20, 15 against
// 27).  Used where the operands carry errors of that size themselves; differences of nodal
// values take the accurate sum.
__host__ __device__ __forceinline__ df add_q(df a, df b) {
  const df s = df_two_sum(a.hi, b.hi);
  return df_fast_two_sum(s.hi, s.lo + (a.lo + b.lo));
}
__host__ __device__ __forceinline__ df sub_q(df a, df b) { return add_q(a, -b); }
__host__ __device__ __forceinline__ df fma_q(df a, df b, df c) {
  const df p = df_two_prod(a.hi, b.hi);
  const float pl = fmaf(a.hi, b.lo, fmaf(a.lo, b.hi, p.lo));
  const df s = df_two_sum(p.hi, c.hi);
  return df_fast_two_sum(s.hi, s.lo + (pl + c.lo));
}

// x * p for a power of two p (exact: both parts scale; half the cost of a product)
__host__ __device__ __forceinline__ df mul_pow2(df x, float p) { return df(x.hi * p, x.lo * p); }
__host__ __device__ __forceinline__ float mul_pow2(float x, float p) { return x * p; }
__host__ __device__ __forceinline__ double mul_pow2(double x, double p) { return x * p; }

// Split of a loaded double and back, by integer and FP32 operations.  GB300 converts between
// double and float on its FP64 pipe, two lanes per clock and SM: one conversion takes as long
// as 64 FP32 operations.  The element kernels split 8 to 12 loaded doubles per lane and
// join 3 or 4; with conversions (and a DADD per split) that alone held the FP64 pipe for 656
// clocks per warp.  Values outside float's normal range (below 2^-126, above its largest,
// infinities, NaN) take the conversions.
union df_bits32 { float f; uint32_t u; };
union df_bits64 { double d; uint64_t u; };
__host__ __device__ __forceinline__ uint32_t df_f2u(float f) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(f);
#else
  df_bits32 b; b.f = f; return b.u;
#endif
}
__host__ __device__ __forceinline__ float df_u2f(uint32_t u) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(u);
#else
  df_bits32 b; b.u = u; return b.f;
#endif
}
__host__ __device__ __forceinline__ uint64_t df_d2u(double d) {
#ifdef __CUDA_ARCH__
  return (uint64_t)__double_as_longlong(d);
#else
  df_bits64 b; b.d = d; return b.u;
#endif
}
__host__ __device__ __forceinline__ double df_u2d(uint64_t u) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)u);
#else
  df_bits64 b; b.u = u; return b.d;
#endif
}

// hi = x rounded to float, lo = the remainder rounded to float (as two conversions and a
// subtraction would give, but for the rounding of the last bit of lo): the leading 24 bits
// by moving the mantissa, the other 29 as two floats of 23 and 6 bits read off a mantissa
// under x's exponent, then one Fast2Sum rounds hi to nearest.
__host__ __device__ __forceinline__ df df_split(double x) {
  const uint64_t b = df_d2u(x);
  const uint32_t w1 = (uint32_t)(b >> 32), w0 = (uint32_t)b;
  const uint32_t m = (w1 & 0x7fffffffu) - (896u << 20);  // exponent rebased to float's
  if (m - (1u << 20) >= (254u << 20)) {                  // not a normal float
    if (((w1 & 0x7fffffffu) | w0) == 0u) return df(0.0f, 0.0f);
    const float h = (float)x;
    return df(h, (float)(x - (double)h));
  }
  const uint32_t t = (w1 & 0x80000000u) | (m << 3) | (w0 >> 29);
  const uint32_t e = t & 0xff800000u, r = w0 & 0x1fffffffu;
  const float one = df_u2f(e);  // x's sign and power of two
  const float l1 = (df_u2f(e | (r >> 6)) - one) * 1.1920928955078125e-07f;                 // 2^-23
  const float l2 = (df_u2f(e | ((r & 63u) << 17)) - one) * 1.4210854715202004e-14f;        // 2^-46
  const df s = df_fast_two_sum(df_u2f(t), l1);
  return df_fast_two_sum(s.hi, s.lo + l2);
}
// the double equal to a float
__host__ __device__ __forceinline__ double df_widen(float f) {
  const uint32_t b = df_f2u(f), m = b & 0x7fffffffu;
  if (m - 0x00800000u >= 0x7f000000u && m != 0u) return (double)f;  // denormal, infinity, NaN
  const uint32_t w1 = (b & 0x80000000u) | (m ? (m >> 3) + 0x38000000u : 0u);
  return df_u2d(((uint64_t)w1 << 32) | (uint32_t)(b << 29));
}
__host__ __device__ __forceinline__ double df_to_double(df a) { return df_widen(a.hi) + df_widen(a.lo); }
