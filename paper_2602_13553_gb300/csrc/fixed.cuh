// fixed.cuh -- normal-mode transforms of FP64 rows in 64-bit fixed point.
//
// The FP64 pipe issues one warp instruction every 64 clocks per SM partition
// (two FMAs a clock and SM, measured), the integer pipe a 32 x 32 -> 64
// multiply-add every 2.2 (58 a clock and SM): a sum of products is therefore
// taken in integers, with more bits than FP64 keeps.
//
// A row x_0 .. x_{P-1} is scaled by the power of two above its largest element,
// |x_j| <= 2^ex, and rounded to X_j = x_j 2^(55 - ex).  The mode matrix is
// scaled by the power of two above its largest element, 2^em, and rounded to
// 55 bits likewise (on the host).  Both are split into two signed 28-bit limbs,
// X = X_h 2^28 + X_l, |X_l| <= 2^27, and
//   sum M X = 2^56 sum M_h X_h + 2^28 sum (M_h X_l + M_l X_h) + [sum M_l X_l],
// the last term (2^-55 of the first's scale, zero mean) being dropped: three
// multiply-adds a product, all exact.  Rows folded by the parity of the modes
// (|u| <= 2^56, at most 66 terms) keep every accumulator below 2^62.
//
// Error against the exact sum, in units of 2^ex max|M|: about 2^-57 sqrt(n)
// for n terms (rounding of X and M, the dropped term), then one rounding to 64
// bits at 2^-55 and one to FP64; the FP64 sum it replaces has 2^-54 of a partial
// sum at each of its n additions.
#pragma once

#include <cuda_runtime.h>

namespace pimd {

constexpr int kFixBits = 55;       // |X|, |M| <= 2^55
constexpr int kFixMinE = 128;      // rows below 2^-894 are taken as that
constexpr int kFixMaxE = 2000;     // rows above 2^978, infinite or NaN come out as NaN

// Pairs of terms of a folded sum: even modes (and beads) j <= P/2, rounded up.
__host__ __device__ constexpr int fix_pairs(int P) { return (P / 2 + 2) / 2; }

__device__ __forceinline__ int exp_field(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// round(x 2^(55 - ex)) with ex = E - 1022, E the row's largest exponent field.
__device__ __forceinline__ long long to_fixed(double x, int E) {
  const int hi = __double2hiint(x);
  const int s = min(E - ((hi >> 20) & 0x7ff), 63);
  unsigned long long m =
      ((unsigned long long)(unsigned)((hi & 0xfffff) | 0x100000) << 32) | (unsigned)__double2loint(x);
  m = (((m << 3) >> s) + 1) >> 1;
  return hi < 0 ? -(long long)m : (long long)m;
}

__device__ __forceinline__ int2 fix_limbs(long long u) {
  const long long r = u + 0x8000000;
  return make_int2((int)(r >> 28), (int)(r & 0xfffffff) - 0x8000000);
}

// Accumulators of one sum, and its value in units of 2^(ex + em - 55).
struct FixSum {
  long long h = 0, c = 0;
  // two terms: x = (X_h, X_l) of both, m = (M_h, M_l) of both
  __device__ __forceinline__ void add2(const int4 &x, const int4 &m) {
    h += (long long)x.x * m.x;
    c += (long long)x.x * m.y;
    c += (long long)x.y * m.x;
    h += (long long)x.z * m.z;
    c += (long long)x.z * m.w;
    c += (long long)x.w * m.z;
  }
  __device__ __forceinline__ long long value() const { return (h << 1) + ((c + (1 << 26)) >> 27); }
};

// S 2^(E - 1022 + em - 55) as FP64, NaN for a row that is not finite.
__device__ __forceinline__ double from_fixed(long long S, int E, int em) {
  if (E > kFixMaxE) return __longlong_as_double(0x7ff8000000000000ll);
  if (S == 0) return 0.0;
  const double d = (double)S;
  return __hiloint2double(__double2hiint(d) + ((E - 1022 + em - kFixBits) << 20), __double2loint(d));
}

}  // namespace pimd
