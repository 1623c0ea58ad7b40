// sums.cu -- the two parts of a step that couple all atoms of a system: the
// BZP barostat's B_W (App. E) and fixcom (Sec. III.C), FP64.
//
// Both reduce over every (atom, component) row of P beads.  A lane group (the
// smallest power of two of lanes that holds min(P, 32) beads) takes one row at
// a time, its beads adjacent (coalesced); the groups are spread over many
// blocks, each of which leaves one row of partial sums, and the last block to
// finish (threadfence and count, no waiting) adds the rows in block order and
// does the scalar work.  A group strides the rows by a multiple of three, so
// it always holds the same component.  Every order is fixed by the sizes.
//
// What bounds them is latency: the work is one read of x, v~, F from L2.  As
// single blocks with one thread per atom (strided reads, N P serial terms)
// they were most of a step: the barostat 72 us a call (two a step) for 125
// molecules x 16 beads, fixcom 50 us for 91 molecules x 17 beads and 192 us
// for 100 molecules x 12 Cartesian beads; now 12.0, 10.1 and 9.5.  (The factor
// (e^a - e^-a) / (2 v_W) from the series of sinh would need no division and no
// cancellation, but leaves the published form by its 1e-11 at small a.)
#include "common.cuh"

#include <algorithm>

namespace pimd {

constexpr int kSumThreads = 256;

__device__ __forceinline__ double warp_sum(double v) { return group_sum(v, 32); }

// True in every thread of the block that finishes last; the others' partial
// sums are then visible to it.  Resets the counter for the next launch.
__device__ __forceinline__ bool last_block(unsigned *count) {
  __shared__ bool last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(count, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return false;
  __threadfence();
  if (threadIdx.x == 0) *count = 0;
  return true;
}

// B_W of the BZP barostat (App. E) over [t0, t0 + tB] of the kick that the
// next kernel applies to the current velocities, with n = P.  Isotropic:
//   v_W += (3 tB / W)[n V P_CV - n V P_ext + n kB T] + (tB^2 / W) sum F~0.v~0
//          + (tB^3 / 3W) sum |F~0|^2 / m~0,
//   3 n V P_CV = sum m~0 |v~0|^2 - sum (r - r_c).F + sum_k Tr Xi^(k);
// anisotropic, for each edge a in the mask, the same with the a components
// alone, W the per-edge mass and 3 n V P_CV -> n V P_CV^aa (the Xi_aa rows).
// Then, if a step follows, its v_W at the first A, after O_W (PILE_L: each
// edge its own deviate) and the box after both A sub-steps.
//
// Partial row of a block: [q][c] for q = m v0^2, F0 v0, F0^2 / m, (r - r_c) F,
// virial (isotropic: c = 0 alone).
constexpr int kBaroCols = 15;

__global__ void __launch_bounds__(kSumThreads) k_baro_kick(BaroArgs a) {
  __shared__ double sg[4][kSumThreads];
  __shared__ double sv[3][kSumThreads / 32];
  __shared__ double tot[kBaroCols];
  __shared__ double noise[3];
  const int P = a.P, W = row_lanes(P), gpb = kSumThreads / W;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int lg = threadIdx.x / W, l = threadIdx.x - lg * W;   // group in block, lane in group
  const int g = blockIdx.x * gpb + lg;
  const int S = (int)gridDim.x * gpb / 3 * 3;
  const int rows = a.N * 3;
  const double rp = a.rsp;   // F~0 = (M F)_0 = sum_j F_j / sqrt(P)
  double mv2 = 0.0, fv = 0.0, f2m = 0.0, rcf = 0.0;
  // every lane of a warp runs the same rounds (the shuffles need them all)
  for (int r0 = 0; r0 < rows; r0 += S) {
    const int r = r0 + g;
    const bool on = g < S && r < rows;
    const size_t row = (size_t)r * P;
    double x[4], f[4], sx = 0.0, sf = 0.0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int j = l + q * W;
      const bool h = on && j < P;
      x[q] = h ? a.x[row + j] : 0.0;
      f[q] = h ? a.F[row + j] : 0.0;
      sx += x[q];
      sf += f[q];
    }
    const double mm = on ? a.mass_mm[r / 3] : 1.0, im = on ? a.inv_mm[r / 3] : 1.0;
    const double v = on ? a.v[row] - (a.fix_u ? a.fix_u[r % 3] : 0.0) : 0.0;
    const double xm = group_sum(sx, W) * a.invP;
    const double f0 = rp * group_sum(sf, W);
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (l + q * W < P) rcf = fma(x[q] - xm, f[q], rcf);
    if (l == 0 && on) {
      const double fm = f0 * im;
      const double v0 = fma(a.t0, fm, v);   // at t0 into the kick
      mv2 = fma(mm * v0, v0, mv2);
      fv = fma(f0, v0, fv);
      f2m = fma(f0, fm, f2m);
    }
  }
  rcf = group_sum(rcf, W);
  if (l == 0) {
    sg[0][lg] = mv2;
    sg[1][lg] = fv;
    sg[2][lg] = f2m;
    sg[3][lg] = rcf;
  }
  double vir[3] = {0.0, 0.0, 0.0};
  for (int t = blockIdx.x * kSumThreads + threadIdx.x; t < a.nmol * P; t += gridDim.x * kSumThreads) {
    if (a.axes) {
#pragma unroll
      for (int c = 0; c < 3; ++c) vir[c] += a.W3part[(size_t)t * 3 + c];
    } else {
      vir[0] += a.Wpart[t];
    }
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    if (c == 0 || a.axes) vir[c] = warp_sum(vir[c]);
    if (lane == 0) sv[c][warp] = vir[c];
  }
  __syncthreads();
  if (threadIdx.x < kBaroCols) {
    const int q = threadIdx.x / 3, c = threadIdx.x % 3;
    double s = 0.0;
    if (q < 4) {
      for (int b = 0; b < gpb; ++b)
        if ((blockIdx.x * gpb + b) % 3 == c) s += sg[q][b];
    } else {
      for (int b = 0; b < kSumThreads / 32; ++b) s += sv[c][b];
    }
    a.part[blockIdx.x * kBaroCols + threadIdx.x] = s;
  }
  if (!last_block(a.count)) return;
  // the state the scalar work starts from, requested before the sums
  double *b = a.baro;
  const double V = b[kBaroL] * b[kBaroL + 1] * b[kBaroL + 2], L = b[kBaroL + threadIdx.x % 3];
  double vW = b[kBaroV + threadIdx.x % 3];
  const uint64_t step = (uint64_t)*a.step;
  // the rows of partials: one warp per column
  for (int col = warp; col < kBaroCols; col += kSumThreads / 32) {
    double s = 0.0;
    for (int r = lane; r < (int)gridDim.x; r += 32) s += __ldcg(a.part + r * kBaroCols + col);
    s = warp_sum(s);
    if (lane == 0) tot[col] = s;
  }
  // O_W's deviates: Philox atom 0xffffffff, stream 3, mode 0 (the O of BAOAB,
  // the first O(h/2) of OBABO) or 1 (the second, of the step just completed).
  // The last warp (one column): a lane for each radius and angle
  if (a.thermo && threadIdx.x >= kSumThreads - 32 && (a.step_follows || a.obabo)) {
    const uint4 w = noise_words(a.seed, 0xffffffffu, a.step_follows ? 0u : 1u, 3u, a.step_follows ? step : step - 1);
    uint64_t radius = 0;
    int64_t sn = 0, cs = 0;
    if (lane == 0 || lane == 2) radius = bm_radius_fix(lane ? w.z : w.x);
    if (lane == 1 || lane == 3) bm_angle_fix(lane == 1 ? w.y : w.w, sn, cs);
    const int64_t c1 = __shfl_sync(0xffffffffu, cs, 1), s1 = __shfl_sync(0xffffffffu, sn, 1);
    const int64_t c3 = __shfl_sync(0xffffffffu, cs, 3);
    const uint64_t r0 = __shfl_sync(0xffffffffu, radius, 0), r2 = __shfl_sync(0xffffffffu, radius, 2);
    if (lane < 3) noise[lane] = bm_deviate(lane == 2 ? r2 : r0, lane == 0 ? c1 : (lane == 1 ? s1 : c3));
  }
  __syncthreads();
  // the scalar work, one warp: lane = (edge c, sign of the exponent, which A);
  // the lanes of an edge do the same up to their exponential (isotropic: all do)
  if (threadIdx.x >= 12) return;
  const int c = threadIdx.x % 3, sgn = threadIdx.x / 3 % 2, h = threadIdx.x / 6;
  const double *mv = tot, *sfv = tot + 3, *sf2 = tot + 6, *srcf = tot + 9, *svir = tot + 12;
  const bool moves = !a.axes || (a.axes >> c & 1);
  const double eta = a.axes ? noise[c] : noise[0];
  // O_W: v_W <- c1 v_W + sigW eta; each edge its own deviate, the isotropic
  // v_W the first
  auto langevin = [&](double w) { return moves ? a.c1W * w + a.sigW * eta : w; };
  if (a.obabo && a.step_follows && a.thermo) vW = langevin(vW);   // this step's first O(h/2)
  if (!moves) {
    vW = 0.0;
  } else if (a.axes) {
    vW += a.k1 * (mv[c] - srcf[c] + svir[c] - V * a.npext + a.nkT) + a.k2 * sfv[c] + a.k3 * sf2[c];
  } else {
    vW += a.k1 * ((mv[0] + mv[1] + mv[2] - (srcf[0] + srcf[1] + srcf[2]) + svir[0]) * (1.0 / 3.0) - V * a.npext +
                  a.nkT) +
          a.k2 * (sfv[0] + sfv[1] + sfv[2]) + a.k3 * (sf2[0] + sf2[1] + sf2[2]);
  }
  if (!a.step_follows) {
    // OBABO: the closing O(h/2) of the step just completed (the counter has
    // already been advanced past it)
    if (a.obabo && a.thermo) vW = langevin(vW);
    if (threadIdx.x < 3) b[kBaroV + c] = vW;
    return;
  }
  double vO = vW;
  if (a.thermo && !a.obabo) vO = langevin(vO);
  // the A factors of the centroid mode at v_W (h = 0) and, BAOAB, at v_O (h = 1)
  const double w = h ? vO : vW, x = a.tA * w;
  const double ex = exp(sgn ? -x : x);
  const double other = __shfl_sync(0xfffu, ex, (threadIdx.x + 3) % 12);   // sgn 0: the lane's e^-x
  const double grow2 = __shfl_sync(0xfffu, ex, (threadIdx.x + 6) % 12);   // h 0: e^x of the second A
  if (sgn == 0) {
    double *f = b + (h ? kBaroA2 : kBaroA1) + 3 * c;
    f[0] = ex;
    f[1] = other;
    f[2] = fabs(x) < 1e-8 ? a.tA * (1.0 + x * x / 6.0) : (ex - other) / (2.0 * w);
  }
  if (threadIdx.x >= 3) return;
  b[kBaroVA1 + c] = vW;
  b[kBaroVA2 + c] = vO;
  b[kBaroV + c] = vO;
  // BAOAB: A(h/2) at v_W, O_W, A(h/2) at v_O; OBABO: one A(h) at v_W
  const double Ln = a.obabo ? L * ex : L * ex * grow2;
  b[kBaroL + c] = Ln;
  b[kBaroInvL + c] = 1.0 / Ln;
  if (!(Ln > a.Lmin)) atomicOr(a.err, kErrBoxSmall);
}

// fixcom: the mass-weighted mean velocity u of the centroid mode (normal
// modes, nb = 1) or of every bead (Cartesian, nb = P) as it will stand after
// the closing B(h/2) (and O(h/2)) that the next kernel applies; that kernel
// subtracts u when it loads v.  Partial row of a block: [q][c][k] for
// q = m v, F, m (2 x_k - x_{k-1} - x_{k+1}) (Cartesian: the springs, from the
// small differences), m sigv eta (OBABO's closing O(h/2)).
__global__ void __launch_bounds__(kSumThreads) k_fixcom_f64(FixcomArgs a) {
  __shared__ double sh[4 * 1024];   // [q][group][k]; then the totals [q][c][k]
  const int P = a.P, W = row_lanes(P), gpb = kSumThreads / W;
  const int lg = threadIdx.x / W, l = threadIdx.x - lg * W;
  const int g = blockIdx.x * gpb + lg;
  const int S = (int)gridDim.x * gpb / 3 * 3;
  const int rows = a.N * 3;
  const int nb = a.method == 0 ? 1 : P;
  const uint64_t s = (uint64_t)(*a.step - 1);
  double pv[4] = {0.0, 0.0, 0.0, 0.0}, pf[4] = {0.0, 0.0, 0.0, 0.0};
  double px[4] = {0.0, 0.0, 0.0, 0.0}, pn[4] = {0.0, 0.0, 0.0, 0.0};
  for (int r = g; g < S && r < rows; r += S) {
    const int i = r / 3, c = r - 3 * i;
    const size_t row = (size_t)r * P;
    const double mm = a.mass_mm[i];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int k = l + q * W;
      if (k >= P) continue;
      pf[q] += a.F[row + k];
      if (k >= nb) continue;
      pv[q] = fma(mm, a.v[row + k], pv[q]);
      if (a.method == 1) {
        const double xk = a.x[row + k];
        const double xm = a.x[row + (k == 0 ? P - 1 : k - 1)], xp = a.x[row + (k == P - 1 ? 0 : k + 1)];
        px[q] = fma(mm, (xk - xm) + (xk - xp), px[q]);
      }
      if (a.obabo_thermo)
        pn[q] = fma(mm * a.sigv[i], gauss1(a.seed, (uint32_t)i, (uint32_t)k, kStreamO2, s, c), pn[q]);
    }
  }
  if (a.method == 0) {   // F~_0 sqrt(P) = sum over the beads
    pf[0] = group_sum(pf[0] + pf[1] + pf[2] + pf[3], W);
  }
  const int gs = gpb * nb;   // groups x beads
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int k = l + q * W;
    if (k >= nb) continue;
    sh[lg * nb + k] = pv[q];
    sh[gs + lg * nb + k] = pf[q];
    sh[2 * gs + lg * nb + k] = px[q];
    sh[3 * gs + lg * nb + k] = pn[q];
  }
  __syncthreads();
  const int ncol = 12 * nb;   // [q][c][k]
  double *part = a.part + (size_t)blockIdx.x * ncol;
  for (int t = threadIdx.x; t < ncol; t += kSumThreads) {
    const int q = t / (3 * nb), c = t / nb % 3, k = t % nb;
    double sum = 0.0;
    for (int b = 0; b < gpb; ++b)
      if ((blockIdx.x * gpb + b) % 3 == c) sum += sh[q * gs + b * nb + k];
    part[t] = sum;
  }
  if (!last_block(a.count)) return;
  const int rows_p = (int)gridDim.x;
  if (nb == 1) {   // twelve columns: a warp each
    for (int t = threadIdx.x >> 5; t < ncol; t += kSumThreads / 32) {
      double sum = 0.0;
      for (int b = threadIdx.x & 31; b < rows_p; b += 32) sum += __ldcg(a.part + (size_t)b * ncol + t);
      sum = warp_sum(sum);
      if ((threadIdx.x & 31) == 0) sh[t] = sum;
    }
  } else {         // a thread each, four loads in flight and four partial sums
    for (int t = threadIdx.x; t < ncol; t += kSumThreads) {
      double s4[4] = {0.0, 0.0, 0.0, 0.0};
      for (int b = 0; b < rows_p; b += 4) {
        double v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] = b + q < rows_p ? __ldcg(a.part + (size_t)(b + q) * ncol + t) : 0.0;
#pragma unroll
        for (int q = 0; q < 4; ++q) s4[q] += v[q];
      }
      sh[t] = (s4[0] + s4[1]) + (s4[2] + s4[3]);
    }
  }
  __syncthreads();
  for (int kc = threadIdx.x; kc < 3 * nb; kc += kSumThreads) {
    const int c = kc / nb, k = kc % nb;
    double p = sh[kc], f = sh[3 * nb + kc];
    if (a.method == 0)
      f *= a.rsp;   // F~_0
    else
      f = fma(-a.wn2, sh[6 * nb + kc], f);
    // the closing O(h/2) scales by c1 and adds c2 sigv eta: remove its mean too
    if (a.obabo_thermo) p = fma(a.c2[k] / a.c1[k], sh[9 * nb + kc], p);
    a.u[3 * k + c] = fma(a.half * a.imu0, f, p) * a.imsum;
  }
}

// --- host launchers --------------------------------------------------------
// Blocks: enough groups for `per` rows each, at least three (one per
// component), at most 128 (the last block adds one row of partials per block).
static int sum_blocks(int N, int P, int per) {
  const int gpb = kSumThreads / row_lanes(P);
  const int want = (3 * N + gpb * per - 1) / (gpb * per);
  return std::min(128, std::max(want, (2 + gpb) / gpb));
}

// Doubles of partial sums a system's two reductions need at most.
size_t sums_part_doubles(int N, int P, int method) {
  const int nb = method == 0 ? 1 : P;
  return (size_t)sum_blocks(N, P, 1) * std::max(kBaroCols, 12 * nb);
}

cudaError_t launch_baro_kick(const BaroArgs &a, cudaStream_t s) {
  k_baro_kick<<<sum_blocks(a.N, a.P, 1), kSumThreads, 0, s>>>(a);
  return cudaGetLastError();
}

// One row per group where the rows carry noise (some 70 FP64 operations an
// element); four otherwise, so that the last block adds fewer rows.
cudaError_t launch_fixcom(const FixcomArgs &a, cudaStream_t s) {
  k_fixcom_f64<<<sum_blocks(a.N, a.P, a.obabo_thermo ? 1 : 4), kSumThreads, 0, s>>>(a);
  return cudaGetLastError();
}

}  // namespace pimd
