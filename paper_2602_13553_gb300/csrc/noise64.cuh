// noise64.cuh -- Box-Muller deviates of 32-bit words to FP64 accuracy on the
// integer pipe.
//
// u = (w + 1/2) 2^-32 of a Philox word gives the radius sqrt(-2 ln u) or the
// angle 2 pi u.  An FP64 instruction costs a warp 64 clocks, an integer one
// about 2.2, so logarithm, square root, sine and cosine are taken in 64-bit
// fixed point, table and short polynomial each (the table-driven scheme of
// P. T. P. Tang, ACM TOMS 16, 378 (1990), with the polynomials of log1p, sin
// and cos, here in fixed point), and only the finished deviate becomes FP64.
// "Qn" below is a number with n fraction bits.
//
// Against quadruple precision (every table interval, the extreme words and
// random ones, seven million in all): the radius is within 2^-53.9 (at small radii;
// 2^-56.2 from 1/2 up), sine and cosine within 2^-56.3, and the deviates' rms error is 6e-17,
// FP64 rounding included, against 3e-16 for FP64 log, sqrt and cos of 2 pi u.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace pimd {

struct NoiseLog { int64_t T; uint32_t c, pad; };    // ln c (+ ln 2 in the upper half) Q62, c Q16 ~ 1 / interval
struct NoiseArc { int64_t C, S; };                  // cosine and sine of the interval's centre, Q62

struct NoiseTables {
  NoiseLog log[256];
  NoiseArc arc[256];
};

namespace noise_detail {
typedef __int128 i128;

// ln(p / q) Q62 for p / q in (1/3, 3): 2 atanh((p - q) / (p + q)) by its series, Q90
constexpr int64_t ln_ratio(int64_t p, int64_t q) {
  const i128 a = p - q, b = p + q;
  i128 term = ((i128)1 << 90) * a / b, sum = 0;
  for (int k = 1; term != 0 && k < 200; k += 2) {
    sum += term / k;
    term = term * a / b;
    term = term * a / b;
  }
  return (int64_t)((sum + ((i128)1 << 26)) >> 27);   // 2 sum, Q90 -> Q62
}

constexpr int64_t kLn2 = ln_ratio(2, 1);             // Q62

// sine (odd = 1) or cosine of pi n / 1024, n in (0, 512), by Taylor's series, Q60
constexpr int64_t arc_value(int n, int odd) {
  const i128 pi = 0x3243F6A8885A308D;                // Q60
  const i128 th = pi * n / 1024, th2 = (th * th) >> 60;
  i128 term = odd ? th : (i128)1 << 60, sum = 0;
  for (int k = odd; term != 0 && k < 60; k += 2) {
    sum += term;
    term = -((term * th2) >> 60) / ((k + 1) * (k + 2));
  }
  return (int64_t)(sum << 2);                        // Q62
}

constexpr NoiseTables make_tables() {
  NoiseTables t{};
  for (int j = 0; j < 256; ++j) {
    // interval [1 + j / 256, 1 + (j + 1) / 256): c next to 1 / its centre, and
    // exactly 1/2 in the last, where u -> 1 must give ln u -> 0
    const int64_t den = 512 + 2 * j + 1;
    const int64_t c = j == 255 ? 32768 : (65536 * 512 * 2 + den) / (2 * den);
    t.log[j].c = (uint32_t)c;
    t.log[j].T = ln_ratio(c, 65536) + (j >= 106 ? kLn2 : 0);
    t.arc[j].C = arc_value(2 * j + 1, 0);
    t.arc[j].S = arc_value(2 * j + 1, 1);
  }
  t.log[255].T = 0;
  return t;
}
}  // namespace noise_detail

static __device__ const NoiseTables kNoise = noise_detail::make_tables();

#ifdef __CUDA_ARCH__
#define PIMD_UMULHI64(a, b) __umul64hi(a, b)
#define PIMD_NOISE (&kNoise)
#else   // the same arithmetic on the host, for checking it there
#define PIMD_UMULHI64(a, b) ((uint64_t)(((unsigned __int128)(a) * (b)) >> 64))
static const NoiseTables kNoiseHost = noise_detail::make_tables();
#define PIMD_NOISE (&kNoiseHost)
#endif

// s32(a b / 2^32), u32(a b / 2^32)
__host__ __device__ __forceinline__ int mulhi_s32(int a, int b) { return (int)(((long long)a * b) >> 32); }
__host__ __device__ __forceinline__ uint32_t mulhi_u32(uint32_t a, uint32_t b) {
  return (uint32_t)(((unsigned long long)a * b) >> 32);
}
__host__ __device__ __forceinline__ float rsqrt_seed(float x) {
#ifdef __CUDA_ARCH__
  return rsqrtf(x);
#else
  return 1.0f / sqrtf(x);
#endif
}

// leading zeros of y > 0; 2^e for a normal exponent
__host__ __device__ __forceinline__ int lead_zeros(uint64_t y) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)y);
#else
  return __builtin_clzll(y);
#endif
}
__host__ __device__ __forceinline__ float pow2f(int e) {
#ifdef __CUDA_ARCH__
  return __int_as_float((e + 127) << 23);
#else
  return ldexpf(1.0f, e);
#endif
}

// sqrt(-2 ln u), Q60.
__host__ __device__ __forceinline__ uint64_t bm_radius_fix(uint32_t w) {
  // n = 2 w + 1 = (2^32 + f) 2^-lz, u = n 2^-33: -ln u = a ln 2 + T_j - log1p(r)
  // with r = (1 + f 2^-32) c_j - 1 exact in Q48, |r| < 2^-8.9, and a = lz + 1,
  // or lz in the upper half, whose T_j holds the other ln 2
  const uint64_t n = 2 * (uint64_t)w + 1;
#ifdef __CUDA_ARCH__
  const int lz = w >> 31 ? 0 : 1 + __clz((int)(2 * w + 1));
#else
  const int lz = w >> 31 ? 0 : 1 + __builtin_clz(2 * w + 1);
#endif
  const uint32_t f = (uint32_t)(n << lz);
  const uint32_t j = f >> 24;
  const NoiseLog t = PIMD_NOISE->log[j];
  const int a = lz + (j < 106 ? 1 : 0);
  const int64_t r = (int64_t)(((uint64_t)t.c << 32) + (uint64_t)f * t.c) - ((int64_t)1 << 48);
  // log1p(r) = r - r^2 h, h = 1/2 - r p, p = 1/3 - r (1/4 - r (1/5 - r / 6))
  const int ri = (int)(r >> 9);   // Q39
  const int t1 = 429496730 - (mulhi_s32(ri, 357913941) >> 7);   // Q31
  const int t2 = 536870912 - (mulhi_s32(ri, t1) >> 7);
  const int p = 715827883 - (mulhi_s32(ri, t2) >> 7);
  const uint64_t h = (uint64_t)(((int64_t)1 << 61) - (((int64_t)ri * p) >> 8));   // Q62
  const uint64_t ra = (uint64_t)(r < 0 ? -r : r) << 24;                         // Q72
  const uint64_t r2 = PIMD_UMULHI64(ra, ra);                                    // Q80
  const int64_t l1p = (r << 14) - (int64_t)((PIMD_UMULHI64(r2, h) + 0x8000) >> 16);
  const int64_t tail = t.T - l1p;                                               // Q62
  // near u = 1 (T = 0, a = 0) -ln u itself is small: there the radius needs
  // the tail's own leading bits, from the same series in FP64
  if (a == 0 && j == 255) {
    const double rd = (double)r * 3.552713678800501e-15;   // 2^-48
    double s = 1.0 / 7.0;
    s = 1.0 / 6.0 - rd * s;
    s = 0.2 - rd * s;
    s = 0.25 - rd * s;
    s = 1.0 / 3.0 - rd * s;
    s = 0.5 - rd * s;
    return (uint64_t)(sqrt(-2.0 * (rd - rd * rd * s)) * 1152921504606846976.0);
  }
  const uint64_t y = (uint64_t)(a * (noise_detail::kLn2 >> 4) + (tail >> 4));   // -ln u, Q58
  // s = sqrt(t), t = 2 y (y as Q57): FP32 seed, then two corrections
  // s += (t - s^2) / (2 s) whose residuals are exact
  // (from 32 bits each: a 64-bit conversion takes a slot of the FP64 pipe; the
  // step of 20011 x 17 oscillator beads, OBABO, took 81 us with them, 76.5 so)
  const int nz = lead_zeros(y);
  const float tf = (float)(uint32_t)((y << nz) >> 32) * pow2f(-25 - nz);         // 2^-57 y
  const float rs = rsqrt_seed(tf);
  const uint32_t g0 = (uint32_t)(tf * rs * 268435456.0f);                    // Q28
  const int64_t e0 = (int64_t)(y - (((uint64_t)g0 * g0) << 1));              // Q57, below 2^42
  const float hr = 0.5f * rs;
  const int64_t g1 = ((int64_t)g0 << 22) + (int)((float)(int)(e0 >> 12) * hr * 32.0f);   // Q50: 2^(12 + 50 - 57)
  const int64_t e1 = (int64_t)((y << 43) - (uint64_t)g1 * (uint64_t)g1);      // Q100, below 2^62
  return (uint64_t)((g1 << 10) + (int)((float)(int)(e1 >> 32) * hr * 0.00390625f));   // Q60: 2^(32 + 60 - 100)
}

// sine and cosine of 2 pi u, Q62.
__host__ __device__ __forceinline__ void bm_angle_fix(uint32_t w, int64_t &sn, int64_t &cs) {
  // quadrant, one of 256 intervals of it, and the offset t from the interval's
  // centre in units of 2^-33 of a turn: delta = 2 pi t 2^-33, |delta| < 2^-8.3
  const NoiseArc c = PIMD_NOISE->arc[(w >> 22) & 0xff];
  const int t = (int)(2 * (w & 0x3fffff) + 1) - (1 << 22);
  const uint32_t s = (uint32_t)(t < 0 ? -t : t);
  const uint64_t d = (uint64_t)s * 3373259426u + (((uint64_t)s * 560513589u) >> 32);   // |delta| Q62: 2 pi 2^29
  const uint32_t d32 = (uint32_t)(d >> 22);              // Q40
  const uint32_t z = mulhi_u32(d32, d32);                // delta^2 Q48
  const uint32_t z2 = mulhi_u32(z, z);                   // delta^4 Q64
  // sin = delta (1 - g), g = delta^2 / 6 - delta^4 / 120 (Q50)
  const uint32_t g = mulhi_u32(z, 0xAAAAAAABu) - mulhi_u32(z2, 2185u);
  const uint64_t sd = d - (((uint64_t)d32 * g) >> 28);   // Q62
  // 1 - cos = delta^2 / 2 - delta^4 / 24, Q80: (2 pi)^2 2^-67 t^2, and z2 2^16 / 24
  const uint64_t t2 = (uint64_t)s * s;
  const uint64_t cm = PIMD_UMULHI64(t2 << 19, 11378879155978302162ull) - (((uint64_t)z2 * 178956971u) >> 16);
  const uint64_t C = (uint64_t)c.C, S = (uint64_t)c.S;
  const int64_t sC = (int64_t)(PIMD_UMULHI64(C, sd << 8) >> 6), sS = (int64_t)(PIMD_UMULHI64(S, sd << 8) >> 6);
  const int64_t cc = c.C - (int64_t)(PIMD_UMULHI64(C, cm) >> 16) + (t < 0 ? sS : -sS);
  const int64_t ss = c.S - (int64_t)(PIMD_UMULHI64(S, cm) >> 16) + (t < 0 ? -sC : sC);
  const uint32_t quad = w >> 30;
  const int64_t co = quad & 1 ? ss : cc, si = quad & 1 ? cc : ss;
  cs = quad == 1 || quad == 2 ? -co : co;
  sn = quad >= 2 ? -si : si;
}

// radius (Q60) times sine or cosine (Q62), the deviate as FP64
__host__ __device__ __forceinline__ double bm_deviate(uint64_t radius, int64_t trig) {
  const uint64_t m = (uint64_t)(trig < 0 ? -trig : trig);
  const int64_t e = (int64_t)PIMD_UMULHI64(radius, m << 1);   // Q59
  const double d = (double)(trig < 0 ? -e : e);
#ifdef __CUDA_ARCH__
  return e ? __hiloint2double(__double2hiint(d) - (59 << 20), __double2loint(d)) : 0.0;
#else
  return d * 1.734723475976807e-18;   // 2^-59
#endif
}

}  // namespace pimd
