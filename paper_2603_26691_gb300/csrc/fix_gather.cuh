// FP64 trilinear interpolation on the integer pipe.
//
// GB300 issues one FP64 instruction per warp and scheduler in 64 cycles, and integer instructions in one or
// two, so an FP64 kernel pays for its FP64 instructions and little else.  The field is therefore also kept as
// integers (FixCell, 32 bytes per cell, exact): each component a signed 59-bit mantissa of two limbs of 31 and
// 28 bits beside a biased exponent counted in units of 3 bits, so that most stencils share one exponent per component.
// The eight weights are 58-bit integers built with five multiplications and differences, so that they add up to one
// exactly, and each component's sum is 24 products of limbs with 64-bit accumulation.  The eight products of low limbs
// are not formed: what they would add, two mantissa units at most, is estimated from the mantissas' low limbs and the
// mean of the weights' (dot8).  That leaves the sum without a bias and within a mantissa unit of the exact one, where
// FP64 rounds at four units or more, so a uniform field comes out exactly.  (With 29-bit limbs the products
// are four times as large and cannot be left out: a pass of ten steps of 3e7 particles on 128^3 took 22.2 ms with all
// 32 formed, against 21.1 ms so, and 20.7 ms without them or an estimate, low by a quarter of 2^-53 at worst.)
// Corners of smaller exponents are shifted to the largest one, rounded down: what they lose lies below 2^-55 of the
// largest corner, where an FP64 interpolation rounds at 2^-53 three times.  In units of 2^-53 of the largest corner the
// errors' root mean square is 0.19 for corners of one size (three FP64 lerps: 0.46) and 0.11 for corners over three decades
// (0.25), their mean below 0.001 and -0.02.  (Rounding the shifts to nearest as well takes that mean away, and 4.5 % more
// time.)
#pragma once

#include <cmath>

#include "st_common.cuh"

namespace st {
namespace fix {

constexpr int kLimb = 28;
constexpr int kFrac = 58;                              // weights: 2^58 = 1
constexpr int64_t kOne = int64_t(1) << kFrac;
constexpr int64_t kLimbMask = (int64_t(1) << kLimb) - 1;
constexpr int kExpBias = 6 + 1075;                     // a mantissa of exponent e counts 2^(3 e - kExpBias)

// one cell: a = {x high, x low, y high, y low}, b = {z high, z low, three 10-bit exponents, 0}
struct alignas(32) FixCell {
  int4 a, b;
};

// v = mantissa * 2^(3 e - kExpBias), exact: the FP64 significand shifted by 3 to 5 bits
__device__ __forceinline__ int64_t split(double v, int& e) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  int be = (int)((b >> 52) & 0x7ff);
  int64_t man = (int64_t)(b & 0xfffffffffffffull);
  if (be != 0) man |= int64_t(1) << 52;
  else be = 1;
  e = man == 0 ? 0 : be / 3 + 1;
  if (man) man <<= 6 - (3 * e - be);
  return (b >> 63) ? -man : man;
}
__device__ __forceinline__ FixCell make_cell(double x, double y, double z) {
  int ex, ey, ez;
  const int64_t mx = split(x, ex), my = split(y, ey), mz = split(z, ez);
  FixCell c;
  c.a = make_int4((int)(mx >> kLimb), (int)(mx & kLimbMask), (int)(my >> kLimb), (int)(my & kLimbMask));
  c.b = make_int4((int)(mz >> kLimb), (int)(mz & kLimbMask), ex | (ey << 10) | (ez << 20), 0);
  return c;
}
__device__ __forceinline__ FixCell load_cell(const FixCell* p) {
  FixCell c;
  c.a = __ldg(&p->a);
  c.b = __ldg(&p->b);
  return c;
}

// floor(s 2^(53 + k)) for 0 <= s 2^k <= 1024 (anything else, NaN included: 0)
__device__ __forceinline__ int64_t to_fixed53(double s, int k) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(s);
  const int sh = 1033 - k - (int)(b >> 52);  // negative values have the sign bit up here: sh < 0
  const unsigned long long m = (b << 11) | 0x8000000000000000ull;
  return (unsigned)sh > 63u ? 0 : (int64_t)min(m >> sh, 0x7fffffffffffffffull);
}

// v * 2^ex rounded to FP64.  (The rare results outside the normal numbers out of line: the adjoint converts twelve
// times a step, and its 2e6 particles on 64^3, 40 steps, take 21.9 ms instead of 23.0 ms in the smaller loop.)
static __device__ __noinline__ double to_f64_slow(int64_t v, int ex) { return ldexp((double)v, ex); }
__device__ __forceinline__ double to_f64(int64_t v, int ex) {
  if (v == 0) return 0.0;
  const unsigned long long m = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
  const int lz = __clzll((long long)m);
  const int be = 1023 + 63 - lz + ex;
  if (__builtin_expect((unsigned)(be - 1) >= 2045u, 0)) return to_f64_slow(v, ex);
  const unsigned long long t = m << lz;
  unsigned long long r = ((unsigned long long)(be - 1) << 52) + (t >> 11) + ((t >> 10) & 1ull);
  r |= v < 0 ? 0x8000000000000000ull : 0ull;
  return __longlong_as_double((long long)r);
}

// a b / 2^58, rounded to nearest up to a quarter (the product of the low limbs is not formed)
__device__ __forceinline__ int64_t mul58(int64_t a, int64_t b) {
  const int ah = (int)(a >> kLimb), al = (int)(a & kLimbMask), bh = (int)(b >> kLimb), bl = (int)(b & kLimbMask);
  const int64_t high = (int64_t)ah * bh + (((int64_t)ah * bl + (int64_t)al * bh) >> kLimb);  // in quarters
  return (high + 2) >> (kFrac - 2 * kLimb);
}

// the stencil of a position: base and next cell per axis (periodic), fractions of 2^58, containing cell
struct Stencil {
  int i0[3], i1[3], c0[3];
  int64_t f[3];
};
// Cells per length: a factor, or its binary logarithm where all three are powers of two from 1 to 1024 (then the
// product is exact and only moves the exponent: three FP64 instructions less).
struct Scale {
  double inv_h[3];
  int exact, log2[3];
};
inline Scale make_scale(const double (&inv_h)[3]) {
  Scale s;
  s.exact = 1;
  for (int q = 0; q < 3; ++q) {
    int e = 0;
    s.inv_h[q] = inv_h[q];
    const double m = std::frexp(inv_h[q], &e);
    s.log2[q] = e - 1;
    if (m != 0.5 || e < 1 || e > 11) s.exact = 0;
  }
  return s;
}
__device__ __forceinline__ Stencil stencil(const double (&x)[3], const Scale& sc, const int (&n3)[3]) {
  Stencil st;
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const int64_t S = sc.exact ? to_fixed53(x[q], sc.log2[q]) : to_fixed53(x[q] * sc.inv_h[q], 0);
    st.c0[q] = min((int)(S >> 53), n3[q] - 1);
    const int64_t T = S - (int64_t(1) << 52);  // cell centres lie at halves
    const int ii = min((int)(T >> 53), n3[q] - 1);
    st.f[q] = (T & ((int64_t(1) << 53) - 1)) << (kFrac - 53);
    st.i0[q] = ii < 0 ? ii + n3[q] : ii;
    st.i1[q] = ii + 1 >= n3[q] ? ii + 1 - n3[q] : ii + 1;
  }
  return st;
}

// the weights of the corners k = dx + 2 dy + 4 dz; they add up to kOne (one that would be zero may come out as -1)
__device__ __forceinline__ void weights(const int64_t (&f)[3], int64_t (&W)[8]) {
  const int64_t p = mul58(f[0], f[1]);
  const int64_t xy[4] = {kOne - f[0] - f[1] + p, f[0] - p, f[1] - p, p};
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    W[4 + k] = mul58(xy[k], f[2]);
    W[k] = xy[k] - W[4 + k];
  }
}

// mantissas brought to the largest exponent of the eight corners, component by component (word = the corners'
// exponent words; only called where they differ)
__device__ __forceinline__ void align(int (&uh)[8], int (&ul)[8], const int (&word)[8], int q, int& emax) {
  int e = 0;
#pragma unroll
  for (int k = 0; k < 8; ++k) e = max(e, (word[k] >> (10 * q)) & 1023);
  emax = e;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int sh = min(3 * (e - ((word[k] >> (10 * q)) & 1023)), 63);
    const int64_t v = (((int64_t)uh[k] << kLimb) | (int64_t)ul[k]) >> sh;
    uh[k] = (int)(v >> kLimb);
    ul[k] = (int)(v & kLimbMask);
  }
}

// sum_k W_k u_k of one component, rounded to nearest in units of 2^-4 of the mantissa's.  The products of low limbs are
// estimated: the weights' are as good as random, so their mean times the sum of the mantissas' (nothing for a field of
// FP32 values, whose low limbs are zero).
__device__ __forceinline__ int64_t dot8(const int (&wh)[8], const int (&wl)[8], const int (&uh)[8],
                                        const int (&ul)[8]) {
  // |uh| <= 2^30, the wh add up to 2^30 and the low limbs lie below 2^28: |A| <= 2^60, |B| < 2^62
  int64_t A = 0, B = 0;
  uint32_t low = 0;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    A += (int64_t)uh[k] * wh[k];
    B += (int64_t)uh[k] * wl[k];
    B += (int64_t)ul[k] * wh[k];
    low += (uint32_t)ul[k];
  }
  constexpr int sh = kFrac - 4 - kLimb;
  return (A << (2 * kLimb + 4 - kFrac)) + ((B + (int64_t)((low >> 1) + (1u << (sh - 1)))) >> sh);
}

// the eight corners' mantissas in limbs, brought to one exponent per component
struct Corners {
  int uh[3][8], ul[3][8], e[3];
};
__device__ __forceinline__ void load_corners(const FixCell* __restrict__ F, const Stencil& st, int nx, int ny, Corners& u) {
  int word[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int c = ((k & 1) ? st.i1[0] : st.i0[0]) +
                  nx * (((k & 2) ? st.i1[1] : st.i0[1]) + ny * ((k & 4) ? st.i1[2] : st.i0[2]));
    const FixCell v = load_cell(F + c);
    u.uh[0][k] = v.a.x;
    u.ul[0][k] = v.a.y;
    u.uh[1][k] = v.a.z;
    u.ul[1][k] = v.a.w;
    u.uh[2][k] = v.b.x;
    u.ul[2][k] = v.b.y;
    word[k] = v.b.z;
  }
  int differ = 0;
#pragma unroll
  for (int q = 0; q < 3; ++q) u.e[q] = (word[0] >> (10 * q)) & 1023;
#pragma unroll
  for (int k = 1; k < 8; ++k) differ |= word[k] ^ word[0];
#pragma unroll
  for (int q = 0; q < 3; ++q)
    if (differ & (1023 << (10 * q))) align(u.uh[q], u.ul[q], word, q, u.e[q]);
}

// the interpolated value from the corners and their weights
__device__ __forceinline__ void interpolate(const Corners& u, const int64_t (&W)[8], double (&up)[3]) {
  int wh[8], wl[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    wh[k] = (int)(W[k] >> kLimb);
    wl[k] = (int)(W[k] & kLimbMask);
  }
#pragma unroll
  for (int q = 0; q < 3; ++q) up[q] = to_f64(dot8(wh, wl, u.uh[q], u.ul[q]), 3 * u.e[q] - kExpBias - 4);
}

// the derivatives of the interpolated components by the fraction along axis r: the differences along r at the
// four edges, weighted over the other two axes (a and b, in that order the faster bits of an edge's number)
template <int r>
__device__ __forceinline__ void derivative(const Corners& u, const int64_t (&f)[3], double (&g)[3]) {
  constexpr int a = r == 0 ? 1 : 0, b = r == 2 ? 1 : 2;
  const int64_t p = mul58(f[a], f[b]);
  const int64_t w[4] = {kOne - f[a] - f[b] + p, f[a] - p, f[b] - p, p};
  int wh[4], wl[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    wh[k] = (int)(w[k] >> kLimb);
    wl[k] = (int)(w[k] & kLimbMask);
  }
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    constexpr int sh = kFrac - 3 - kLimb;
    int64_t A = 0, B = int64_t(1) << (sh - 1);  // |A| <= 2^61, |B| < 2^62
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int lo = ((k & 1) << a) | ((k >> 1) << b), hi = lo | (1 << r);
      const int dh = u.uh[q][hi] - u.uh[q][lo], dl = u.ul[q][hi] - u.ul[q][lo];
      A += (int64_t)dh * wh[k];
      B += (int64_t)dh * wl[k];
      B += (int64_t)dl * wh[k];
    }
    g[q] = to_f64((A << (2 * kLimb + 3 - kFrac)) + (B >> sh), 3 * u.e[q] - kExpBias - 3);
  }
}

__device__ __forceinline__ void gather(const FixCell* __restrict__ F, const Stencil& st, int nx, int ny, double (&up)[3]) {
  Corners u;
  load_corners(F, st, nx, ny, u);
  int64_t W[8];
  weights(st.f, W);
  interpolate(u, W, up);
}

}  // namespace fix
}  // namespace st
