// fixed.cuh -- FP64 sums in 64-bit integers.
//
// FP64 without the FP64 pipe.  This chip runs 2 FP64 lanes per clock and SM
// (1/64 of FP32; 1.25 TFLOP/s measured), but 32 lanes of 32 x 32 + 64 bit
// integer multiply-adds.  The weighted sum therefore runs in integers that are
// wider than a double's 53 bits:
//  * the differences of a cell's node values to its base node's, exact or rounded
//    once as doubles, become integers X of 61 bits relative to the cell's largest;
//  * the Lagrange weights are formed as integers W = 6 w 2^60 (times 6, so that
//    no division rounds) from the fractional position t, of which every bit is
//    kept;
//  * operands split at bit 32 into signed halves, X = Xh 2^32 + Xl, and a sum of
//    products is sum Wh Xh + (sum Wh Xl + Wl Xh) / 2^32 in units of 2^64: three
//    multiply-adds a term into two 64-bit sums that cannot overflow (|Xh| <= 2^29
//    and |Wh| < 2^31, four terms with sum |w| <= 1.25).  Wl Xl, at most a quarter
//    of a unit, is left out.  Split at the word size, the halves and the result
//    are registers, not shifts;
//  * the sum is the next axis's operand as it stands: an axis scales by
//    6 2^60 / 2^64 and its sum of |weights|, so operands shrink from 2^61 to
//    2^57.7 and the last unit stays below 2^-56 of the largest difference.
// The sum is converted back once, exactly scaled, with one FP64 rounding: its
// error is a few 2^-56 of the largest difference in the cell, where 84 rounded
// FP64 operations leave a few 2^-53 of the partial sums.  That is less wherever the
// partial sums come within 1/8 of the largest difference, as they do on all but a few
// rows of smooth and rough fields; a row whose weights on the large differences are all
// tiny can be off by more than FP64 would be, relative to itself (measured against
// extended precision on smooth plus rough fields, sphere h = 1/24, in units of 2^-53: E u
// 0.51 in the 2-norm where FP64 has 1.28, entries relative to their sum |w||u| 0.57 rms
// against 0.81 but 17 at worst against 4.5; A^T u 1.26 against 1.91, 2.3 rms against 1.3, 299
// at worst against 7.5).  A cell whose
// differences are not finite or whose largest one is below 2^-883 goes through
// plain FP64.
#pragma once

#include <stdint.h>

namespace {  // (internal linkage: the plain path's call then leaves the callers' registers alone)

// signed halves of x = xh 2^32 + xl
__device__ __forceinline__ void halves(long long x, int32_t &xh, int32_t &xl) {
  xl = (int32_t)x;
  xh = (int32_t)((unsigned long long)x >> 32) + (int32_t)((uint32_t)xl >> 31);
}

// cross sums start at half a unit of the word they lose, so that they round
constexpr long long HALF = 0x80000000ll;
__device__ __forceinline__ long long high_word(long long cr) { return (long long)(int32_t)(cr >> 32); }

// a b + c, one instruction
__device__ __forceinline__ long long mad_wide(int32_t a, int32_t b, long long c) {
  long long d;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
  return d;
}

__device__ __forceinline__ void mac(long long &hh, long long &cr, int32_t wh, int32_t wl, int32_t xh, int32_t xl) {
  hh = mad_wide(wh, xh, hh);
  cr = mad_wide(wh, xl, cr);
  cr = mad_wide(wl, xh, cr);
}

// a b / 2^64 to within 1.25 units
__device__ __forceinline__ long long mul_high(long long a, long long b) {
  int32_t ah, al, bh, bl;
  halves(a, ah, al);
  halves(b, bh, bl);
  return mad_wide(ah, bh, high_word(mad_wide(al, bh, mad_wide(ah, bl, HALF))));
}

// 6 2^60 times the Lagrange weights of one axis, in halves.  With tau = t - 1 (exact):
//   cubic      q = tau (tau - 1), P = q tau:
//              6 w = { 2q - P, 3 (P - q - 2 tau + 2), 3 (2 tau - P), P + q }
//   quadratic  6 w = { 3 (tau^2 - tau), 6 (1 - tau^2), 3 (tau^2 + tau) }
template <int NP>
__device__ __forceinline__ void fixed_weights(double t, int32_t (&wh)[4], int32_t (&wl)[4]) {
  const long long b = __double_as_longlong(t);
  const int sh = (int)(b >> 52) - 1023;  // t is in [1/2, 2] up to rounding: sh in -2 .. 1
  long long t60 = (long long)(((b & 0xFFFFFFFFFFFFFll) | 0x10000000000000ll) << 8);
  t60 = (sh >= 0) ? (t60 << sh) : (t60 >> min(-sh, 62));
  const long long one = 1ll << 60, tau = t60 - one;
  long long w[4];
  if constexpr (NP == 4) {
    const long long q = mul_high(tau << 2, (tau - one) << 2);  // 2^62 x 2^62 -> 2^60
    const long long P = mul_high(q << 2, tau << 2);
    const long long c = P - 2 * tau;
    w[0] = 2 * q - P;
    w[1] = 3 * (c - q + 2 * one);
    w[2] = -3 * c;
    w[3] = P + q;
  } else {
    const long long s = mul_high(tau << 2, tau << 2);
    w[0] = 3 * (s - tau);
    w[1] = 6 * (one - s);
    w[2] = 3 * (s + tau);
    w[3] = 0;
  }
#pragma unroll
  for (int k = 0; k < NP; ++k) halves(w[k], wh[k], wl[k]);
}

// ordering key of |d|: its high word, with a bit for a denormal whose bits are
// all in the low one
__device__ __forceinline__ unsigned fx_key(double d) {
  return ((unsigned)__double2hiint(d) & 0x7FFFFFFFu) | (unsigned)(__double2loint(d) != 0);
}

// a set of values whose largest key is `top` has an exponent the integers serve
// (finite, and no scale factor leaves the normal range), or is all zero
__device__ __forceinline__ bool fx_ok(unsigned top) {
  const int em = (int)(top >> 20);
  return em < 2040 && (em >= 140 || top == 0u);
}

// d as an integer in units of 2^(em - 1075 - K), em the largest exponent field of
// the set: |result| < 2^(53 + K)
__device__ __forceinline__ long long fx_of(double d, int em, int K) {
  const int hi = __double2hiint(d);
  const int e = (hi >> 20) & 0x7FF;
  unsigned long long m =
      ((unsigned long long)(((unsigned)hi & 0xFFFFFu) | 0x100000u) << 32) | (unsigned)__double2loint(d);
  m = (e == 0) ? 0ull : ((m << K) >> min(em - e, 63));
  return (hi < 0) ? -(long long)m : (long long)m;
}

// c 2^k for a normal c and result: the exponent field moved
__device__ __forceinline__ double fx_scale(double c, int k) {
  return __hiloint2double(__double2hiint(c) + k * (1 << 20), __double2loint(c));
}

// what a cell's sum over DIM axes (operands fx_of(d, em, 8)) is multiplied with;
// negative where the cell needs plain FP64.  512/27 and 64/9 both lie half a unit
// above the double next to them, 2^-54 of themselves, which scaled_sum adds.
template <int DIM>
__device__ __forceinline__ double fx_cell_scale(unsigned top) {
  constexpr double back = (DIM == 3) ? 4096.0 / 216.0 : 256.0 / 36.0;  // every axis multiplied by 6 / 16
  if (!fx_ok(top)) return -1.0;
  return (top == 0u) ? 1.0 : fx_scale(back, (int)(top >> 20) - 1083);
}

// sc z + b, z with the scale's missing half unit
__device__ __forceinline__ double scaled_sum(double sc, long long z, double b) {
  return fma(sc, (double)(z + (z >> 54)), b);
}

// E u - u_c of one row in plain FP64 (the rare cells outside the integer range)
template <int DIM, int NP>
__device__ __noinline__ double slow_row(const double *t, const int2 *ln, int split, const double *u, int64_t ld,
                                        double uc) {
  double wx[4], wy[4], wz[4];
  cpm_lagrange<NP, double>(t[0], wx);
  cpm_lagrange<NP, double>(t[1], wy);
  if (DIM == 3) cpm_lagrange<NP, double>(t[2], wz);
  else { wz[0] = 1.0; wz[1] = wz[2] = wz[3] = 0.0; }
  double acc = 0.0;
  for (int cz = 0; cz < ((DIM == 3) ? NP : 1); ++cz)
    for (int cy = 0; cy < NP; ++cy) {
      const int2 se = ln[cz * 4 + cy];
      for (int cx = 0; cx < NP; ++cx) {
        const int32_t idx = (cx < split) ? (se.x + cx) : (se.y + (cx - split));
        acc += (wx[cx] * (wy[cy] * wz[cz])) * (u[(int64_t)idx * ld] - uc);
      }
    }
  return acc;
}

}  // namespace
