// wide.cuh -- sums of FP64 terms in 128-bit integers.
//
// The FP64 pipe issues one warp instruction every 64 clocks per SM partition,
// and a compensated addition takes seven: ~450 clocks a term.  Here a term's
// 53-bit mantissa is shifted to the scale of the largest term met so far and
// added to a 128-bit integer, some 30 instructions of the integer pipe: bits
// below 2^-101 of the largest term are cut (a compensated chain keeps 2^-106 of
// its partial sums), additions are exact, and 2^26 terms fit.
#pragma once

#include <cuda_runtime.h>

#include "fixed.cuh"

namespace pimd {

struct WideSum {
  static constexpr int kShift = 48;   // bits kept below a term of the largest exponent
  __int128 a;                         // units of 2^(e - 1075 - kShift)
  int e;                              // largest exponent field met

  __device__ __forceinline__ void clear() {
    a = 0;
    e = 0;
  }
  __device__ __forceinline__ void rescale(int E) {
    a >>= min(E - e, 127);
    e = E;
  }
  __device__ __forceinline__ void add(double x) {
    const int hi = __double2hiint(x);
    const int f = (hi >> 20) & 0x7ff;
    const long long m =
        (long long)(((unsigned long long)(unsigned)((hi & 0xfffff) | (f ? 0x100000 : 0)) << 32) |
                    (unsigned)__double2loint(x));
    const int fe = max(f, 1);
    if (fe > e) rescale(fe);
    a += ((__int128)(hi < 0 ? -m : m) << kShift) >> min(e - fe, 127);
  }
  __device__ __forceinline__ void add(const WideSum &o) {
    const int E = max(e, o.e);
    a = (a >> min(E - e, 127)) + (o.a >> min(E - o.e, 127));
    e = E;
  }
  // correctly rounded; NaN once a term was infinite or NaN
  __device__ __forceinline__ double value() const {
    if (e >= 0x7ff) return __longlong_as_double(0x7ff8000000000000ll);
    if (a == 0) return 0.0;
    const unsigned __int128 u = a < 0 ? -(unsigned __int128)a : (unsigned __int128)a;
    const unsigned long long uh = (unsigned long long)(u >> 64);
    const int n = uh ? __clzll((long long)uh) : 64 + __clzll((long long)(unsigned long long)u);
    const unsigned __int128 w = u << n;
    const double d = __ull2double_rn((unsigned long long)(w >> 64) | (unsigned long long)((unsigned long long)w != 0));
    const double r = scalbn(d, e - 1075 - kShift + 64 - n);
    return a < 0 ? -r : r;
  }
  __device__ __forceinline__ WideSum shfl_down(int o) const {
    WideSum w;
    const unsigned __int128 u = (unsigned __int128)a;
    const unsigned long long lo = __shfl_down_sync(0xffffffffu, (unsigned long long)u, o);
    const unsigned long long hi = __shfl_down_sync(0xffffffffu, (unsigned long long)(u >> 64), o);
    w.a = (__int128)(((unsigned __int128)hi << 64) | lo);
    w.e = __shfl_down_sync(0xffffffffu, e, o);
    return w;
  }
};

// Warp-wide sum (all lanes call); lane 0 holds the total.
__device__ __forceinline__ WideSum warp_wide(WideSum v) {
  v.rescale(__reduce_max_sync(0xffffffffu, v.e));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v.a += v.shfl_down(o).a;
  return v;
}

}  // namespace pimd
