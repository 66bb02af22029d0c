// lane_ops.cuh -- lane-group Q1 arithmetic shared by the element kernels: 2^d lanes of a
// warp hold the corners of one element and the Gauss points next to them.  Interpolation
// is a tensor product of 1D operators on the two nodes of an axis: at the Gauss point
// next to node b (xi = -g for b = 0, +g for b = 1, g = 1/sqrt 3)
//     value:       a u_b + b' u_{1-b} = u_b - b' (u_b - u_{1-b}),   a = (1 + g)/2, b' = (1 - g)/2
//     derivative:  (u_1 - u_0) / h           (constant along the axis)
// applied axis by axis with the partner value fetched by a lane shuffle (lane ^ 2^k).
// The test side (element vector r_c = w sum_q [N_c(q) S_q + grad N_c(q) . Phi_q], w =
// (h/2)^d) is the transpose: the value operator is symmetric and the derivative's
// transpose sends s_b (x_0 + x_1) / h to node b (s_0 = -1, s_1 = +1).
#pragma once

#include <cstdint>

#include "df32.cuh"

namespace {

constexpr double kG = 0.57735026918962576450914878050196;  // 1/sqrt(3)
constexpr unsigned kFull = 0xffffffffu;

template <typename T>
__device__ __forceinline__ T flip(T x, int k) {
  return __shfl_xor_sync(kFull, x, 1 << k);
}
__device__ __forceinline__ df flip(df x, int k) {
  return df(__shfl_xor_sync(kFull, x.hi, 1 << k), __shfl_xor_sync(kFull, x.lo, 1 << k));
}

// value and gradient at this lane's Gauss point from this lane's nodal value x
// (nb = -b': the value operator is x - b' (x - partner))
template <typename T, int D>
__device__ __forceinline__ void interp_vg(T x, T nb, const T (&sh)[3], T& val, T (&g)[3]) {
  T I = x;
#pragma unroll
  for (int k = 0; k < D; ++k) {
    const T pI = flip(I, k);
    T pG[3];
#pragma unroll
    for (int j = 0; j < k; ++j) pG[j] = flip(g[j], k);
#pragma unroll
    for (int j = 0; j < k; ++j) g[j] = fma(nb, g[j] - pG[j], g[j]);
    const T d = I - pI;
    g[k] = sh[k] * d;
    I = fma(nb, d, I);
  }
#pragma unroll
  for (int k = D; k < 3; ++k) g[k] = T(0);
  val = I;
}

template <typename T, int D>
__device__ __forceinline__ void interp_g(T x, T nb, const T (&sh)[3], T (&g)[3]) {
  T I = x;
#pragma unroll
  for (int k = 0; k < D; ++k) {
    const T pI = flip(I, k);
    T pG[3];
#pragma unroll
    for (int j = 0; j < k; ++j) pG[j] = flip(g[j], k);
#pragma unroll
    for (int j = 0; j < k; ++j) g[j] = fma(nb, g[j] - pG[j], g[j]);
    const T d = I - pI;
    g[k] = sh[k] * d;
    if (k + 1 < D) I = fma(nb, d, I);
  }
#pragma unroll
  for (int k = D; k < 3; ++k) g[k] = T(0);
}

template <typename T, int D>
__device__ __forceinline__ T interp_v(T x, T nb) {
#pragma unroll
  for (int k = 0; k < D; ++k) x = fma(nb, x - flip(x, k), x);
  return x;
}

// ---- pairs -----------------------------------------------------------------------
// Two scalars that go through the same operations (the two species, two velocity
// components, two test rows) as one value.  For FP32 and double-float the pair's
// operations are GB300's packed ones (add / mul / fma .f32x2: two lanes' work in one issue
// slot, the same rounding): the FP32 pipe does no more per clock, but the instruction
// count halves.  That is what the double-float kernels were short of: 3,700 instructions
// straight through per warp (59 KB) left their warps waiting for instruction fetches
// (stall no_instruction 4.3 of 11 cycles per issue, FMA pipe at 61 %).
using ::fma;
struct f2 {
  float2 v;
};
__device__ __forceinline__ f2 operator+(f2 a, f2 b) { return {__fadd2_rn(a.v, b.v)}; }
__device__ __forceinline__ f2 operator*(f2 a, f2 b) { return {__fmul2_rn(a.v, b.v)}; }
__device__ __forceinline__ f2 fma(f2 a, f2 b, f2 c) { return {__ffma2_rn(a.v, b.v, c.v)}; }
__device__ __forceinline__ f2 operator-(f2 a, f2 b) { return {__ffma2_rn(b.v, make_float2(-1.f, -1.f), a.v)}; }
struct d2 {
  double x, y;
};
__device__ __forceinline__ d2 operator+(d2 a, d2 b) { return {a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ d2 operator-(d2 a, d2 b) { return {a.x - b.x, a.y - b.y}; }
__device__ __forceinline__ d2 operator*(d2 a, d2 b) { return {a.x * b.x, a.y * b.y}; }
__device__ __forceinline__ d2 fma(d2 a, d2 b, d2 c) { return {fma(a.x, b.x, c.x), fma(a.y, b.y, c.y)}; }
// two double-floats, each with the operations of df32.cuh
struct df2 {
  f2 hi, lo;
};
__device__ __forceinline__ df2 df2_two_sum(f2 a, f2 b) {
  const f2 s = a + b;
  const f2 bb = s - a;
  return {s, (a - (s - bb)) + (b - bb)};
}
__device__ __forceinline__ df2 df2_fast_two_sum(f2 a, f2 b) {
  const f2 s = a + b;
  return {s, b - (s - a)};
}
__device__ __forceinline__ df2 operator+(df2 a, df2 b) {
  df2 s = df2_two_sum(a.hi, b.hi);
  const df2 t = df2_two_sum(a.lo, b.lo);
  s = df2_fast_two_sum(s.hi, s.lo + t.hi);
  return df2_fast_two_sum(s.hi, s.lo + t.lo);
}
// a - b with the signs of b in the sums
__device__ __forceinline__ df2 operator-(df2 a, df2 b) {
  const f2 s = a.hi - b.hi, sb = s - a.hi;                     // s = a + (-b), sb its share of -b
  const f2 e = (a.hi - (s - sb)) - (b.hi + sb);
  const f2 t = a.lo - b.lo, tb = t - a.lo;
  const f2 f = (a.lo - (t - tb)) - (b.lo + tb);
  const df2 r = df2_fast_two_sum(s, e + t);
  return df2_fast_two_sum(r.hi, r.lo + f);
}
__device__ __forceinline__ df2 operator*(df2 a, df2 b) {
  const f2 p = a.hi * b.hi;
  const f2 e = fma(a.hi, b.hi, f2{make_float2(-p.v.x, -p.v.y)});
  return df2_fast_two_sum(p, fma(a.hi, b.lo, fma(a.lo, b.hi, e)));
}
__device__ __forceinline__ df2 fma(df2 a, df2 b, df2 c) { return a * b + c; }
// the quick forms of df32.cuh; for the other types the plain operations
__device__ __forceinline__ df2 add_q(df2 a, df2 b) {
  const df2 s = df2_two_sum(a.hi, b.hi);
  return df2_fast_two_sum(s.hi, s.lo + (a.lo + b.lo));
}
__device__ __forceinline__ df2 sub_q(df2 a, df2 b) {
  const f2 s = a.hi - b.hi, sb = s - a.hi;
  return df2_fast_two_sum(s, ((a.hi - (s - sb)) - (b.hi + sb)) + (a.lo - b.lo));
}
__device__ __forceinline__ df2 fma_q(df2 a, df2 b, df2 c) {
  const f2 p = a.hi * b.hi;
  const f2 pl = fma(a.hi, b.lo, fma(a.lo, b.hi, fma(a.hi, b.hi, f2{make_float2(-p.v.x, -p.v.y)})));
  const df2 s = df2_two_sum(p, c.hi);
  return df2_fast_two_sum(s.hi, s.lo + (pl + c.lo));
}
using ::add_q;
using ::fma_q;
using ::sub_q;
#define PLAIN_Q(T)                                                             \
  __device__ __forceinline__ T add_q(T a, T b) { return a + b; }               \
  __device__ __forceinline__ T sub_q(T a, T b) { return a - b; }               \
  __device__ __forceinline__ T fma_q(T a, T b, T c) { return fma(a, b, c); }
PLAIN_Q(float)
PLAIN_Q(double)
PLAIN_Q(f2)
PLAIN_Q(d2)
#undef PLAIN_Q

template <typename C>
struct PairOf;
template <>
struct PairOf<float> {
  using type = f2;
};
template <>
struct PairOf<double> {
  using type = d2;
};
template <>
struct PairOf<df> {
  using type = df2;
};
template <typename C>
using pair_t = typename PairOf<C>::type;
__device__ __forceinline__ f2 pair(float a, float b) { return {make_float2(a, b)}; }
__device__ __forceinline__ d2 pair(double a, double b) { return {a, b}; }
__device__ __forceinline__ df2 pair(df a, df b) { return {pair(a.hi, b.hi), pair(a.lo, b.lo)}; }
template <typename C>
__device__ __forceinline__ pair_t<C> both(C a) { return pair(a, a); }
__device__ __forceinline__ float first(f2 a) { return a.v.x; }
__device__ __forceinline__ float second(f2 a) { return a.v.y; }
__device__ __forceinline__ double first(d2 a) { return a.x; }
__device__ __forceinline__ double second(d2 a) { return a.y; }
__device__ __forceinline__ df first(df2 a) { return df(a.hi.v.x, a.lo.v.x); }
__device__ __forceinline__ df second(df2 a) { return df(a.hi.v.y, a.lo.v.y); }
__device__ __forceinline__ f2 flip(f2 a, int k) { return pair(flip(a.v.x, k), flip(a.v.y, k)); }
__device__ __forceinline__ d2 flip(d2 a, int k) { return {flip(a.x, k), flip(a.y, k)}; }
__device__ __forceinline__ df2 flip(df2 a, int k) { return {flip(a.hi, k), flip(a.lo, k)}; }

// ---- the same operators with their constant factors taken out --------------------
// With rho = b' / a = 2 - sqrt 3 the value operator is a (u_b + rho u_{1-b}): one fused
// multiply-add per axis where u_b - b' (u_b - u_{1-b}) needs a subtraction as well.  The
// factors a gather in front: a value is a^D times the scaled value computed here, a
// derivative a^(D-1) / h times the scaled one.  Derivatives are kept reflected, s_k d_k u
// with s_k = +1 on the lanes of node 1 of the axis and -1 on those of node 0: the scaled
// reflected derivative is u_b - u_{1-b} without a sign, products of two gradients are the
// same in reflected components, and the transposed derivative of a reflected Phi is
// Phi - partner.  A contraction with a plain vector reflects that vector (reflect()).
// In double-float the differences and the values they are taken of use the accurate
// operations, everything else the quick ones: against 64 bits that is as exact as accurate
// operations throughout (relative error of the residual on the membrane-band octree
// 1.58e-14 both ways, 1.72e-14 with FP64-style interpolation in accurate operations; with
// quick differences 1.70e-14).
constexpr double kVal = 0.5 * (1.0 + kG);                 // a
// b' / a = 2 - sqrt 3, rounded once: it acts on every axis of the interpolation and of the
// tests the same way, so its error adds up (written as (1 - kG) / (1 + kG) it was one unit in
// the last place off, and the FP64 J V 1.4 times as far from 64 bits)
constexpr double kRho = 0.26794919243112270647255365849413;
__host__ __device__ constexpr double ipow(double x, int n) { return n <= 0 ? 1.0 : x * ipow(x, n - 1); }

template <typename T, int D>
__device__ __forceinline__ T lane_v(T x, T rho) {
#pragma unroll
  for (int k = 0; k < D; ++k) x = fma_q(rho, flip(x, k), x);
  return x;
}
// scaled reflected gradient (D components); the scaled value too when VAL
template <typename T, int D, bool VAL>
__device__ __forceinline__ void lane_vg(T x, T rho, T& val, T (&g)[3]) {
  T I = x;
#pragma unroll
  for (int k = 0; k < D; ++k) {
    const T pI = flip(I, k);
    T pG[3];
#pragma unroll
    for (int j = 0; j < k; ++j) pG[j] = flip(g[j], k);
#pragma unroll
    for (int j = 0; j < k; ++j) g[j] = fma_q(rho, pG[j], g[j]);
    g[k] = I - pI;
    if (VAL || k + 1 < D) I = fma(rho, pI, I);
  }
  if (VAL) val = I;
}
// transpose: node contribution / a^D of the tests S and reflected Phi, Phi in units of a / h
template <typename T, int D>
__device__ __forceinline__ T lane_test(T S, T (&Phi)[3], T rho) {
  T A = S;
#pragma unroll
  for (int k = D - 1; k >= 0; --k) {
    const T pA = flip(A, k);
    const T pH = flip(Phi[k], k);
    T pP[3];
#pragma unroll
    for (int j = 0; j < k; ++j) pP[j] = flip(Phi[j], k);
    A = add_q(fma_q(rho, pA, A), sub_q(Phi[k], pH));
#pragma unroll
    for (int j = 0; j < k; ++j) Phi[j] = fma_q(rho, pP[j], Phi[j]);
  }
  return A;
}
// s_k x for lane corner c: the sign bit flipped on the lanes of node 0 of axis k
__device__ __forceinline__ uint32_t reflect_mask(int c, int k) { return ((unsigned)~c << (31 - k)) & 0x80000000u; }
__device__ __forceinline__ float reflect(float x, uint32_t m) { return __uint_as_float(__float_as_uint(x) ^ m); }
__device__ __forceinline__ double reflect(double x, uint32_t m) {
  return __hiloint2double(__double2hiint(x) ^ (int)m, __double2loint(x));
}
__device__ __forceinline__ df reflect(df x, uint32_t m) { return df(reflect(x.hi, m), reflect(x.lo, m)); }

// 2^e exactly, from the exponent bits (|e| well inside the exponent range)
__device__ __forceinline__ float pow2i(int e, float) { return __int_as_float((127 + e) << 23); }
__device__ __forceinline__ double pow2i(int e, double) {
  return __longlong_as_double((long long)(1023 + e) << 52);
}
// c 2^e for a positive constant c, by its exponent bits (no FP64 instruction)
__device__ __forceinline__ float const_pow2(double c, int e, float) {
  return __int_as_float(__float_as_int((float)c) + (e << 23));
}
__device__ __forceinline__ double const_pow2(double c, int e, double) {
  return __hiloint2double(__double2hiint(c) + (e << 20), __double2loint(c));
}
__device__ __forceinline__ df const_pow2(double c, int e, df) { return mul_pow2(df(c), pow2i(e, 0.0f)); }
// x c 2^e.  In FP32 the constant is two floats (a rounded constant would be a factor on a
// whole term: a^2 is 4e-8 off, as much as all other rounding of the FP32 kernels together).
// The low part's product goes into the fused operation of the high part, which then rounds
// once; the other way round two roundings of the whole value meet.
__host__ __device__ __forceinline__ float times_const_f(float x, double c, int e) {
  const float h = (float)c, p = df_u2f((uint32_t)(127 + e) << 23);
  return fmaf(x, h * p, x * ((float)(c - (double)h) * p));
}
template <typename C>
__device__ __forceinline__ C times_const(C x, double c, int e) {
  return x * const_pow2(c, e, C(0));
}
template <>
__device__ __forceinline__ float times_const(float x, double c, int e) {
  return times_const_f(x, c, e);
}
__device__ __forceinline__ d2 times_const2(d2 x, double c, int e) { return x * both<double>(const_pow2(c, e, 0.0)); }
__device__ __forceinline__ df2 times_const2(df2 x, double c, int e) { return x * both<df>(const_pow2(c, e, df(0))); }
__device__ __forceinline__ f2 times_const2(f2 x, double c, int e) {
  const float h = (float)c, p = pow2i(e, 0.0f);
  return fma(x, both<float>(h * p), x * both<float>((float)(c - (double)h) * p));
}
// (c x, -c y)
__device__ __forceinline__ d2 times_pm(d2 x, double c) { return x * pair(c, -c); }
__device__ __forceinline__ df2 times_pm(df2 x, double c) { return x * pair(df(c), -df(c)); }
__device__ __forceinline__ f2 times_pm(f2 x, double c) {
  const float h = (float)c, l = (float)(c - (double)h);
  return fma(x, pair(h, -h), x * pair(l, -l));
}
// x 2^e
__device__ __forceinline__ float times_pow2(float x, int e) { return x * pow2i(e, 0.0f); }
__device__ __forceinline__ double times_pow2(double x, int e) { return x * pow2i(e, 0.0); }
__device__ __forceinline__ df times_pow2(df x, int e) { return mul_pow2(x, pow2i(e, 0.0f)); }

// value and gradient of corner i's shape function at this lane's Gauss point (corner c)
template <typename T, int D>
__device__ __forceinline__ void shape_at(int i, int c, T inv_h, T& N, T (&dN)[3]) {
  const T fs = T(0.5 * (1.0 + kG)), fo = T(0.5 * (1.0 - kG));
  T f[3];
#pragma unroll
  for (int k = 0; k < D; ++k) f[k] = (((i ^ c) >> k) & 1) ? fo : fs;
  N = T(1);
#pragma unroll
  for (int k = 0; k < D; ++k) N *= f[k];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    T a = T(0);
    if (k < D) {
      a = ((i >> k) & 1) ? inv_h : -inv_h;
#pragma unroll
      for (int l = 0; l < D; ++l)
        if (l != k) a *= f[l];
    }
    dN[k] = a;
  }
}

// loaded value in the arithmetic type, and back to the storage type
template <typename C, typename T>
__device__ __forceinline__ C to_compute(T x) { return C(x); }
template <>
__device__ __forceinline__ df to_compute<df, double>(double x) { return df_split(x); }
template <typename T>
__device__ __forceinline__ T to_storage(T x) { return x; }
template <typename T>
__device__ __forceinline__ T to_storage(df x) { return df_to_double(x); }

}  // namespace
