// ljfix.cuh -- Lennard-Jones pairs in 64-bit fixed point (FP64 water force).
//
// An FP64 instruction costs a warp 64 clocks, a 64-bit high product 17 and
// a 32-bit multiply-add 2.2, so the pairs of the O-O sum are evaluated in
// integers.  Lengths are scaled by the power of two 2^b above the cutoff and
// x = r^2 / 2^2b; y = 2^-e / x is in (0, 1] down to the distance 2^(b - e/2),
// which lies between 0.56 and 0.79 sigma (farther out for sigma below a tenth of
// the cutoff, where e is at its cap; closer pairs, and systems whose
// scales do not fit, take the FP64 expressions).  With C = 2 (2^e sigma^2 /
// 2^2b)^3 the pair's terms are, per component c,
//   T = y^3 (C y^3 - 1),  f_c = y T d_c / 2^b,
// energy, virial and force being constants times sum (T - y^3), sum T and
// sum f_c.  "Qn" is a number with n fraction bits; sums are 128-bit integers,
// exact and free of order.
//
// Rounding: terms vary by 2^-3e (T) and 2^-4e (f) between the cutoff and the
// closest pair, so each is formed from the reciprocal of the normalised x and
// shifted to the sum's unit: T and f_c keep 2^-55 (at e = 7, 2^-53) or more of
// the pair's own size, where the FP64 expressions round at 2^-53 several times.
// Against 60 decimal digits, pairs from 0.85 of the cutoff on, sigma 3.166, rms
// error of the force over the pair's own, at cutoffs 6, 12 and 20: 1.7e-16,
// 1.8e-16, 1.8e-16 (its rounding to FP64 included); the FP64 expressions 3.9e-16,
// 4.1e-16, 4.1e-16; every term cut at one place, Q58 or Q63, 2.8e-14, 2.0e-13,
// 1.4e-11 (a pass of 512 molecules x 64 beads, 20 steps, took 1.56 ms so; 1.61 now).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <cmath>

namespace pimd {

// Positions and separations have `pos` fraction bits, in angstrom: 53 where every
// edge is below 256 A, 50 below 2048 A.  Of the 2^(63 - pos) A that 64 bits hold a
// quarter is used at set-up and half at run time (the barostat may grow a box; the
// rest is room for the wrap's rounding).  A coordinate of less than 2^(52 - pos) A is
// rounded where FP64 had it exactly: with 50 bits throughout, the force of a pair
// 2.5 to 5.9 A apart in a box of 12.42 A was 5.4e-16 of itself off (rms, from FP64
// positions around the origin), FP64 expressions 5.1e-16; with 53 bits 1.3e-16.
constexpr int kPosFine = 53, kPosCoarse = 50;

struct LjFix {
  int on;                      // 0: every pair in FP64
  int pos;                     // fraction bits of positions and separations
  int b, e;
  double edge;                 // edges from here on take the FP64 expressions
  uint64_t rc2;                // cutoff, x Q64
  uint64_t xmin;               // closer pairs in FP64, x Q62
  uint64_t C;                  // Q58
  float rpre2;                 // 1.008 rc^2 in units of 2^(32 - pos) A squared: the quick test
  double fs, us, ws, w3;       // force, energy (half), virial (half), diagonal virial of the sums
};

inline LjFix lj_fix_setup(double eps, double sig, double rc, const double *box) {
  LjFix p{};
  int b = 0;
  while (std::ldexp(1.0, b) < 1.01 * rc && b < 13) ++b;
  while (b > -10 && std::ldexp(1.0, b - 1) >= 1.01 * rc) --b;
  const double s2 = sig * sig * std::ldexp(1.0, -2 * b);
  int e = 0;
  while (e < 7 && s2 * std::ldexp(1.0, e + 1) <= 3.17) ++e;
  const double ratio = s2 * std::ldexp(1.0, e);
  p.on = ratio <= 3.17 && std::ldexp(1.0, b) >= 1.01 * rc && rc > 0.01;
  p.pos = kPosFine;
  for (int c = 0; c < 3; ++c)
    if (!(box[c] < std::ldexp(1.0, 61 - kPosFine))) p.pos = kPosCoarse;
  for (int c = 0; c < 3; ++c) p.on = p.on && box[c] < std::ldexp(1.0, 61 - p.pos);
  p.edge = std::ldexp(1.0, 62 - p.pos);
  p.b = b;
  p.e = e;
  if (!p.on) return p;
  const double c6 = ratio * ratio * ratio;
  p.rc2 = (uint64_t)std::ldexp(rc * rc, 64 - 2 * b);
  p.xmin = (uint64_t)std::ldexp(1.0 + 1.0 / 1024, 62 - e);
  p.C = (uint64_t)std::ldexp(2.0 * c6, 58);
  p.rpre2 = (float)(1.008 * rc * rc * std::ldexp(1.0, 2 * (p.pos - 32)));
  p.fs = 24.0 * eps * c6 * std::ldexp(1.0, -b - 57 - 3 * e);
  p.w3 = 24.0 * eps * c6 * std::ldexp(1.0, -57 - 3 * e);
  p.us = eps * c6 * std::ldexp(1.0, -59 - 3 * e);
  p.ws = 12.0 * eps * c6 * std::ldexp(1.0, -59 - 3 * e);
  return p;
}

#ifdef __CUDA_ARCH__
#define PIMD_MULHI(a, b) __umul64hi(a, b)
__device__ __forceinline__ float lj_rcp(float x) {   // within one unit in the last place
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
#define PIMD_RCP(x) lj_rcp(x)
#define PIMD_CLZ(x) __clzll((long long)(x))
#define PIMD_FLOAT(bits) __uint_as_float(bits)
#else   // the same arithmetic on the host, for checking it there
#define PIMD_MULHI(a, b) ((uint64_t)(((unsigned __int128)(a) * (b)) >> 64))
#ifndef PIMD_RCP
#define PIMD_RCP(x) (1.0f / (x))
#endif
#define PIMD_CLZ(x) __builtin_clzll(x)
inline float lj_float(uint32_t bits) {
  float f;
  __builtin_memcpy(&f, &bits, 4);
  return f;
}
#define PIMD_FLOAT(bits) lj_float(bits)
#endif

// 1 / (4 X) of X = xn 2^-64 in [1/2, 1), Q64 in (2^62, 2^63], to 2^-61 of
// itself: FP32 seed of the leading 24 bits, then two Newton steps v += v (1 - X v).
// X and v are cut so that each residual, exact modulo 2^64, stays inside it: the
// first is below 2^-21 (24 bits rounded, the seed two units off) of 2^-17, the
// second below 2^-39.6 (v cut to Q40, and the first squared) of 2^-39.
__host__ __device__ __forceinline__ uint64_t lj_recip(uint64_t xn) {
  const float X = PIMD_FLOAT(0x3f000000u + (uint32_t)(((xn >> 39) + 1) >> 1) - 0x800000u);
  const uint32_t v0 = (uint32_t)(PIMD_RCP(X) * 1073741824.0f);                               // Q30
  const int64_t e0 = -(int64_t)((xn >> 14) * v0);                                            // Q80
  const uint64_t v1 =
      ((uint64_t)v0 << 10) + (uint64_t)(((int64_t)(int)(v0 >> 1) * (int)(e0 >> 32)) >> 37);   // Q40
  const int64_t e1 = -(int64_t)((xn >> 2) * v1);                                             // Q102
  return (v1 << 22) + (uint64_t)(((int64_t)(int)(v1 >> 11) * (int)(e1 >> 32)) >> 37);         // Q62
}

// x 2^pos modulo 2^64, rounded (positions are kept wrapped into the box, so the
// modulus never shows).
__host__ __device__ __forceinline__ int64_t fix_pos(double x, int pos) {
#ifdef __CUDA_ARCH__
  const uint64_t bits = (uint64_t)__double_as_longlong(x);
#else
  uint64_t bits;
  __builtin_memcpy(&bits, &x, 8);
#endif
  const int s = (int)((bits >> 52) & 0x7ff) - 1075 + pos;
  const uint64_t m = (bits & 0xfffffffffffffull) | 0x10000000000000ull;
  uint64_t r;
  if (s >= 0)
    r = s < 64 ? m << s : 0;
  else
    r = s > -60 ? ((m >> (-s - 1)) + 1) >> 1 : 0;
  return bits >> 63 ? -(int64_t)r : (int64_t)r;
}

// Position wrapped into the box edge L (its fix_pos LQ): x - L floor(x / L),
// up to one rounding of the quotient either side.
__host__ __device__ __forceinline__ int64_t fix_wrap(double x, int pos, float xf, float invL, int64_t LQ) {
  return fix_pos(x, pos) - (int64_t)floorf(xf * invL) * LQ;
}

// Minimum image of a difference of two wrapped positions.
__host__ __device__ __forceinline__ int64_t fix_mic(int64_t d, int64_t LQ) {
  const int hi = (int)(d >> 32), half = (int)(LQ >> 33);
  if (hi >= half) d -= LQ;
  if (hi < -half) d += LQ;
  return d;
}

struct LjSums {
  __int128 f[3] = {0, 0, 0};          // Q(57 + 4 e)
  __int128 T = 0;                     // Q(59 + 3 e)
  __int128 y3 = 0;                    // Q(58 + 3 e)
  __int128 w[3] = {0, 0, 0};          // f_c d_c (diagonal virial), as f
};

// +-v 2^up, v < 2^63, up < 32
__host__ __device__ __forceinline__ void add_signed(__int128 &s, uint64_t v, bool neg, int up) {
  const int64_t t = neg ? -(int64_t)v : (int64_t)v;
#ifdef __CUDA_ARCH__   // three funnel shifts: a 128-bit shift by a variable is four times that
  const uint32_t lo = (uint32_t)t, hi = (uint32_t)((uint64_t)t >> 32), sg = (uint32_t)((int)hi >> 31);
  const uint64_t a = ((uint64_t)__funnelshift_l(lo, hi, up) << 32) | (lo << up);
  const uint64_t b = ((uint64_t)sg << 32) | __funnelshift_l(hi, sg, up);
  s += (__int128)(((unsigned __int128)b << 64) | a);
#else
  s += (__int128)t * ((__int128)1 << up);
#endif
}

// One pair's terms; d = x_j - x_i minimum image, |d_c| < 2^b.  Returns false
// for a pair closer than the fixed-point range.
template <bool kDiag>
__host__ __device__ __forceinline__ bool lj_fix_pair(const LjFix &p, const int64_t (&d)[3], LjSums &s) {
  const int sh = 64 - p.pos - p.b;   // at least 2: 2^b < 2.02 rc, and rc is below half an edge
  uint64_t dn[3], r2 = 0;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    dn[c] = (uint64_t)(d[c] < 0 ? -d[c] : d[c]) << sh;   // Q64
    r2 += PIMD_MULHI(dn[c], dn[c]);
  }
  if (r2 >= p.rc2) return true;
  if ((r2 >> 2) <= p.xmin) return false;
  // y = 2^-e / x = w 2^(2 - m), w the reciprocal of the normalised x; y < 1 above xmin
  const int nx = PIMD_CLZ(r2), m3 = 3 * (p.e - nx);      // m >= 1
  const uint64_t w = lj_recip(r2 << nx);                 // Q64, (1/4, 1/2]
  const uint64_t w3 = PIMD_MULHI(PIMD_MULHI(w, w), w);   // (1/64, 1/8]
  const uint64_t y3 = m3 > 6 ? w3 >> (m3 - 6) : w3 << (6 - m3);              // Q64
  const uint64_t Cy = PIMD_MULHI(p.C, y3), one = (uint64_t)1 << 58;          // Q58
  const bool neg = Cy < one;
  uint64_t Pm = neg ? one - Cy : Cy - one;                                   // |C y^3 - 1| Q58, below 64
  const int k = Pm >> 59 ? PIMD_CLZ(Pm) : 5, up = 5 - k;
  Pm <<= k;                                                                  // Q(58 + k)
  const uint64_t T = PIMD_MULHI(w3 << 2, Pm), G = PIMD_MULHI(w, T);
  add_signed(s.T, T, neg, 3 * nx + up);
  add_signed(s.y3, w3, false, 3 * nx);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const uint64_t f = PIMD_MULHI(G, dn[c]);
    add_signed(s.f[c], f, neg != (d[c] < 0), 4 * nx + up);
    // x < 2^-nx: the shifted component is still below 1
    if (kDiag) add_signed(s.w[c], PIMD_MULHI(f, dn[c] << (nx >> 1)), neg, 4 * nx + up - (nx >> 1));
  }
  return true;
}

// A sum as FP64, correctly rounded: one conversion of its leading 64 bits.
__host__ __device__ __forceinline__ double fix_sum(__int128 v) {
  const int64_t hi = (int64_t)(v >> 64), lo = (int64_t)v;
  if (hi == lo >> 63) return (double)lo;
  const int n = PIMD_CLZ((uint64_t)(hi ^ (hi >> 63))) - 1;   // spare sign bits; hi is neither 0 nor -1 but for its sign
  const unsigned __int128 u = (unsigned __int128)v << n;
  const double d = (double)((int64_t)(u >> 64) | (int64_t)((uint64_t)u != 0));
#ifdef __CUDA_ARCH__
  return __hiloint2double(__double2hiint(d) + ((64 - n) << 20), __double2loint(d));
#else
  return std::ldexp(d, 64 - n);
#endif
}

// sum (T - y^3) in the units of T.
__host__ __device__ __forceinline__ double fix_energy(const LjSums &s) { return fix_sum(s.T - 2 * s.y3); }

}  // namespace pimd
