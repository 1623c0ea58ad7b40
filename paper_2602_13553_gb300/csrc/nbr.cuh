// nbr.cuh -- O-O neighbour lists on ring-polymer centroids (single systems).
//
// A pair (m, j) can interact at some bead only if its centroid distance at
// the last build was below rc + skin, as long as
//   2 max_m |c_m - c_m(build)| + 2 max_{m,k} |x_O^k - c_m| <= skin
// (triangle inequality on the minimum-image metric: a pair's bead distance
// is at least its build-time centroid distance minus both centroid drifts
// and both bead deviations).  The step kernel writes per-block maxima of the
// two terms and the current centroids; a list is rebuilt when the bound
// exceeds the skin (or when the positions came from outside).
//
// A molecule's list is grouped by bucket (j mod NS), in index order within a
// bucket: the force kernels give buckets to warps, so their sums depend only on
// the interacting pairs and a rebuilt list changes no bit.  One warp lists a
// molecule (a thread each, testing every pair twice in FP64, took 0.75 ms a
// build at 512 molecules).
#pragma once

#include "common.cuh"

namespace pimd {

// Barrier of a block's first `threads` threads (whole warps).
__device__ __forceinline__ void block_part_sync(int threads) {
  asm volatile("bar.sync 1, %0;" ::"r"(threads) : "memory");
}

// Number of neighbours of molecule m within rc + skin, listed by bucket (j mod
// NS) and index, by one warp: FP32 test on the differences of the FP64
// centroids, in FP64 where it is close.
__device__ __forceinline__ int list_molecule(const NbrList &a, const double (&L)[3], const double (&iL)[3], int m,
                                             int NS, int *nl, int *off) {
  const int lane = threadIdx.x & 31;
  const double c0 = a.ccur[3 * m], c1 = a.ccur[3 * m + 1], c2 = a.ccur[3 * m + 2];
  const float rl = (float)a.rlist, lo = rl * rl * (1.0f - 1e-5f), hi = rl * rl * (1.0f + 1e-5f);
  const float Lf[3] = {(float)L[0], (float)L[1], (float)L[2]};
  const float If[3] = {(float)iL[0], (float)iL[1], (float)iL[2]};
  auto near = [&](int j) {
    const double e0 = a.ccur[3 * j] - c0, e1 = a.ccur[3 * j + 1] - c1, e2 = a.ccur[3 * j + 2] - c2;
    const float f0 = fmaf(-rint_mul((float)e0, If[0]), Lf[0], (float)e0);
    const float f1 = fmaf(-rint_mul((float)e1, If[1]), Lf[1], (float)e1);
    const float f2 = fmaf(-rint_mul((float)e2, If[2]), Lf[2], (float)e2);
    const float r2 = f0 * f0 + f1 * f1 + f2 * f2;
    // unwrapped differences of many boxes lose FP32 digits: FP64 there too
    const float far = fmaxf(fmaxf(fabsf((float)e0), fabsf((float)e1)), fabsf((float)e2));
    if (far < 8.0f * rl) {
      if (r2 < lo) return true;
      if (r2 > hi) return false;
    }
    const double d0 = mic(e0, L[0], iL[0]), d1 = mic(e1, L[1], iL[1]), d2 = mic(e2, L[2], iL[2]);
    return d0 * d0 + d1 * d1 + d2 * d2 < a.rlist * a.rlist;
  };
  int total = 0;
  const int n0 = (a.nmol + NS - 1) / NS;   // candidates of bucket 0, the longest
  int seg = 1;                             // lanes per bucket, 32 / seg buckets a round
  while (seg < n0 && seg < 32) seg <<= 1;
  const int sg = lane / seg, tl = lane - sg * seg;
  for (int b = 0; b < NS; b += 32 / seg) {
    const int bb = b + sg;
    for (int t0 = 0; t0 < n0; t0 += seg) {   // more than one round only with a whole warp per bucket
      const int j = bb + (t0 + tl) * NS;
      const bool hit = bb < NS && j < a.nmol && j != m && near(j);
      const unsigned mask = __ballot_sync(0xffffffffu, hit);
      const int pos = total + __popc(mask & ((1u << lane) - 1u));
      if (t0 == 0 && tl == 0 && bb < NS) off[bb] = pos;
      if (hit && pos < kMaxNeighbours) nl[pos] = j;
      total += __popc(mask);
    }
  }
  if (total > kMaxNeighbours) {   // report, and use an empty list
    if (lane == 0) atomicOr(a.err, kErrNbrOverflow);
    __syncwarp();
    for (int b = lane; b < NS; b += 32) off[b] = 0;
    total = -1;
  }
  if (lane == 0) off[NS] = total < 0 ? 0 : total;
  __syncwarp();
  return total;
}

// FP32 at or above a non-negative FP64 value, by its bits (a conversion takes a
// slot of the FP64 pipe).
__device__ __forceinline__ float float_above(double x) {
  const int hi = __double2hiint(x), e = hi >> 20;
  if (e >= 1151) return __int_as_float(0x7f800000);
  if (e < 897) return __int_as_float(0x00800000);
  return __int_as_float((((e - 896) << 23) | ((hi & 0xfffff) << 3) | (int)((unsigned)__double2loint(x) >> 29)) + 1);
}

// This step's rebuild decision from the step kernel's per-block maxima, by the
// first `threads` threads of a block.  Taken in FP32, towards a rebuild: one
// that comes early changes no sum.
__device__ __forceinline__ bool skin_exceeded(const double *blkmax, int n, double skin, int threads) {
  __shared__ longlong2 s_mx[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = threads >> 5;
  // the maxima are non-negative: they compare as integers, off the FP64 pipe
  long long md = 0, me = 0;
  const longlong2 *bm = reinterpret_cast<const longlong2 *>(blkmax);
#pragma unroll 4
  for (int b = threadIdx.x; b < n; b += threads) {
    const longlong2 e = bm[b];
    md = max(md, e.x);
    me = max(me, e.y);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    md = max(md, __shfl_xor_sync(0xffffffffu, md, o));
    me = max(me, __shfl_xor_sync(0xffffffffu, me, o));
  }
  if (lane == 0) s_mx[warp] = make_longlong2(md, me);
  block_part_sync(threads);
  for (int w = 0; w < nw; ++w) {
    const longlong2 e = s_mx[w];
    md = max(md, e.x);
    me = max(me, e.y);
  }
  const float d2 = __fadd_ru(float_above(__longlong_as_double(md)), float_above(__longlong_as_double(me)));
  return d2 >= float_above(skin) * 0.49999985f;
}

__device__ __forceinline__ void list_box(const NbrList &a, double (&L)[3], double (&iL)[3]) {
  const bool db = a.dbox != nullptr;   // the barostat's box: edges, then their inverses
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    L[c] = db ? a.dbox[c] : a.box[c];
    iL[c] = db ? a.dbox[3 + c] : a.invbox[c];
  }
}

// A list built in shared memory kept for the following steps, by one warp.
__device__ __forceinline__ void keep_list(const NbrList &a, int m, int NS, int total, const int *nl, const int *off) {
  const int lane = threadIdx.x & 31;
  for (int e = lane; e < total; e += 32) a.nbr[(size_t)m * kMaxNeighbours + e] = nl[e];
  for (int b = lane; b <= NS; b += 32) a.off[(size_t)m * (NS + 1) + b] = off[b];
  if (lane < 3 && total >= 0) a.cref[3 * m + lane] = a.ccur[3 * m + lane];
}

}  // namespace pimd
