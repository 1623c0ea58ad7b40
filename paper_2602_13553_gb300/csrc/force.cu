// force.cu -- bead-batched forces U(r^(k)) of every bead k in one grid
// (Eq. 1: each bead feels the physical potential of its own copy of the
// system), FP64, plus the per-bead energy U^(k) and virial Tr Xi^(k) that the
// estimators of App. A need.
//
// Harmonic well: thread (atom i, bead k), F = -m mvv2e w^2 x.
// Water-like model: warps over (molecule, chunk of beads); the beads of the
// chunk sit in adjacent lanes, so each lane's gather of a neighbour's bead is
// a contiguous segment of that neighbour's bead row.  O-O Lennard-Jones runs
// over a centroid neighbour list (cutoff + skin) shared by all beads.  Each
// molecule sums its full neighbour list (no atomics), so forces are
// deterministic and independent of what else is on the GPU.
#include <algorithm>

#include "common.cuh"
#include "nbr.cuh"

namespace pimd {

// Per-block bead sums of U and W in a fixed order: the block holds `groups`
// groups of P lanes (one atom or molecule per group).
__device__ __forceinline__ void block_bead_sums(double u, double w, int P, int groups,
                                                double *Upart, double *Wpart) {
  __shared__ double sU[256];
  __shared__ double sW[256];
  sU[threadIdx.x] = u;
  sW[threadIdx.x] = w;
  __syncthreads();
  for (int k = threadIdx.x; k < P; k += blockDim.x) {
    double su = 0.0, sw = 0.0;
    for (int g = 0; g < groups; ++g) {
      su += sU[g * P + k];
      sw += sW[g * P + k];
    }
    Upart[(size_t)blockIdx.x * P + k] = su;
    Wpart[(size_t)blockIdx.x * P + k] = sw;
  }
}

__global__ void __launch_bounds__(256) k_force_harmonic_f64(ForceArgs a) {
  const int P = a.P;
  const int per = blockDim.x / P;                  // atoms per block
  const int i = blockIdx.x * per + threadIdx.x / P;
  const int k = threadIdx.x % P;
  double u = 0.0, w = 0.0;
  if (threadIdx.x < per * P && i < a.N) {
    const double ks = __ldg(a.kspring + i);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const size_t id = ((size_t)i * 3 + d) * P + k;
      const double x = a.x[id];
      const double f = -ks * x;
      a.F[id] = f;
      u = fma(0.5 * ks * x, x, u);
      w = fma(x, f, w);
    }
  }
  const int groups = min(per, a.N - blockIdx.x * per);
  block_bead_sums(u, w, P, groups, a.Upart, a.Wpart);
  if (a.step_inc && blockIdx.x == 0 && threadIdx.x == 0) *a.step_inc += a.inc;
}

// Water-like model, FP64.  A unit of work is one molecule and a chunk of
// Bk = min(P, 32) beads, or G = 32 / Bk molecules where the beads leave lanes
// free: lane = (molecule u of the unit, bead kl), beads in adjacent lanes, so
// a gather of a neighbour's bead row is a contiguous segment.
//
// What bounds it is the FP64 pipe (a warp instruction in 64 clocks per SM
// partition) and, in small systems, the length of one warp's chain:
//  * the O-O pairs run in 64-bit fixed point on the integer pipe (ljfix.cuh),
//    positions from a wrapped fixed-point copy of the oxygens' beads; pairs
//    closer than its range, and systems it does not fit, take the FP64
//    expressions on the FP64 positions;
//  * a system with many units takes them whole, one warp each (split = 1: no
//    reduction, four units to a block); a smaller one splits a unit's neighbour
//    list over `split` warps, which also take the step's list check, and gives
//    its bonds and angle to one more that starts at once; the partial sums are
//    joined as integers, a component to a warp, and converted once.
// Measured, us a launch: 512 molecules x 64 beads 172 in FP64, now 39 (FP64
// instructions 10, integer issue 16 of it); 64 x 32 16.7 and 9.8.  Seven list warps,
// FP64 partial sums and two bonded warps behind the list check, against this form
// (before a pair's terms were formed at its own scale, ljfix.cuh): 64 x 32 beads
// 11.1 / 10.4, 100 x 12 13.2 / 11.1 (11.5 now), 125 x 16 with the diagonal virial
// 16.1 / 13.5 (13.6 now).
// A neighbour's bucket (j mod NS) decides its warp, so every sum depends only on
// the set of interacting pairs: a rebuilt list cannot change a bit.
// kDiag (anisotropic barostat) also sums the diagonal of the virial tensor,
// Xi_aa = sum d_a f_a, into W3part.
struct Bonded {
  double fO[3], fH[2][3], U, W, w3[3];
};

// O-H bonds, U = 1/2 kb (r - r0)^2 each, and the H-O-H angle, U = 1/2 kth
// (theta - th0)^2, of molecule m at bead k.
template <bool kDiag>
__device__ __forceinline__ void bonded_f64(const ForceArgs &a, int m, int k, const double (&L)[3],
                                           const double (&iL)[3], Bonded &o) {
  const int P = a.P;
  const double *x = a.x + (size_t)9 * m * P + k;
  double d[2][3], r2[2], ir[2];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const double xo = x[c * P];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      double e = x[(3 + 3 * h + c) * P] - xo;
      // the minimum image, only where a component reaches half a box (the
      // comparison of high words may fall to either side of a tie, as rint may)
      if ((__double2hiint(e) & 0x7fffffff) >= __double2hiint(L[c]) - 0x100000) e = mic(e, L[c], iL[c]);
      d[h][c] = e;
    }
  }
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    r2[h] = d[h][0] * d[h][0] + d[h][1] * d[h][1] + d[h][2] * d[h][2];
    ir[h] = rsqrt(r2[h]);
  }
  o.U = o.W = 0.0;
  double gd[2], ga;   // H force h: gd[h] d_h + ga d_{1-h}
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    // r - r0 with r = r2 ir corrected by half a Newton step of its square
    const double r = r2[h] * ir[h];
    const double dr = fma(0.5 * ir[h], fma(-r, r, r2[h]), r - a.r0), kd = a.kb * dr;
    o.U = fma(0.5 * kd, dr, o.U);
    gd[h] = -kd * ir[h];
    o.W = fma(gd[h], r2[h], o.W);
  }
  // F_h = kth (theta - th0) / sin(theta) d cos(theta) / d r_h; the virial of
  // an angle is zero (it does not change with the scale)
  const double ir01 = ir[0] * ir[1];
  const double dot = d[0][0] * d[1][0] + d[0][1] * d[1][1] + d[0][2] * d[1][2];
  const double cth = fmin(1.0, fmax(-1.0, dot * ir01));
  const double dth = acos(cth) - a.th0, kd = a.kth * dth;
  o.U = fma(0.5 * kd, dth, o.U);
  const double pref = kd * rsqrt(fma(-cth, cth, 1.0));
  ga = pref * ir01;
#pragma unroll
  for (int h = 0; h < 2; ++h) gd[h] = fma(-pref * cth * ir[h], ir[h], gd[h]);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    o.fH[0][c] = fma(ga, d[1][c], gd[0] * d[0][c]);
    o.fH[1][c] = fma(ga, d[0][c], gd[1] * d[1][c]);
    o.fO[c] = -(o.fH[0][c] + o.fH[1][c]);
    if (kDiag) o.w3[c] = fma(d[1][c], o.fH[1][c], d[0][c] * o.fH[0][c]);
  }
}

// A pair in FP64, from the FP64 positions: forces on i, U, Tr Xi (and Xi_aa).
struct PairF64 {
  double f[3] = {0.0, 0.0, 0.0}, U = 0.0, W = 0.0, w3[3] = {0.0, 0.0, 0.0};
  bool any = false;
};

template <bool kDiag>
__device__ __noinline__ void pair_f64(const ForceArgs &a, const double *L, const double *iL, int m, int j, int k,
                                      PairF64 &s) {
  const int P = a.P;
  const double *xi = a.x + (size_t)9 * m * P + k, *xj = a.x + (size_t)9 * j * P + k;
  double d[3], r2 = 0.0;
  for (int c = 0; c < 3; ++c) {
    d[c] = mic(xj[c * P] - xi[c * P], L[c], iL[c]);
    r2 = fma(d[c], d[c], r2);
  }
  if (!(r2 < a.rc * a.rc)) return;
  s.any = true;
  const double inv = 1.0 / r2;
  const double s2 = a.sig * a.sig * inv;
  const double s6 = s2 * s2 * s2;
  s.U = fma(4.0 * a.eps, fma(s6, s6, -s6), s.U);
  const double fr = 24.0 * a.eps * fma(2.0 * s6, s6, -s6) * inv;   // force on j = fr * d
  for (int c = 0; c < 3; ++c) {
    s.f[c] = fma(-fr, d[c], s.f[c]);
    if (kDiag) s.w3[c] = fma(fr * d[c], d[c], s.w3[c]);
  }
  s.W = fma(fr, r2, s.W);
}

// kSplit: 0 one warp a unit, 1 up to 14 list warps, 2 four of them, with the
// registers (96) that put four blocks on an SM: a pass of 512 molecules x 64
// beads, 20 steps, 1.66 ms with 101 registers and three blocks, 1.56 so (1.61 with
// today's pair terms); five blocks (72, spills) are faster only at 1024 units and more
// (68.7 against 69.5 us a step there, 35.4 against 33.3 at 400)
template <bool kDiag, int kSplit>
__global__ void __launch_bounds__(kSplit == 2 ? 160 : (kSplit ? 480 : 128), kSplit == 2 ? 4 : 1) k_force_water_f64(ForceArgs a, int split) {
  constexpr int NC = kDiag ? 14 : 11;   // F (9), U, Tr Xi, then Xi_xx, Xi_yy, Xi_zz
  extern __shared__ __align__(16) unsigned char fsm[];
  const int P = a.P;
  const int Bk = P < 32 ? P : 32, G = 32 / Bk;
  const int NS = kLJWarps * a.nb.groups;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int unit = kSplit ? blockIdx.x : blockIdx.x * 4 + warp;
  const int role = kSplit ? warp : 0;   // 0 .. split - 1: the list; then bonds and angle
  // chunk by chunk: the warps of an SM gather from one chunk's rows
  const int nmg = (a.nmol + G - 1) / G;
  const int chunk = unit / nmg, mg = unit - chunk * nmg;
  const int u = lane / Bk, kl = lane - u * Bk;
  const int m = mg * G + u, k = chunk * Bk + kl;
  const bool on = u < G && m < a.nmol && k < P;   // (a last block's spare warps have k >= P)
  double L[3], iL[3];
  list_box(a.nb, L, iL);
  // a small system's blocks take the step's rebuild decision themselves (the
  // same one from the same maxima) and list their own molecules in shared
  // memory; the block of chunk 0 also keeps the lists and the new centroids
  int *s_nl = reinterpret_cast<int *>(fsm);             // [G][kMaxNeighbours]
  int *s_off = s_nl + G * kMaxNeighbours;               // [G][NS + 1]
  bool own = false;
  if (kSplit && a.check_nbr && role < split) {
    own = skin_exceeded(a.nb.blkmax, a.nb.nblk_check, a.nb.skin, 32 * split);
    if (own) {
      for (int q = warp; q < G; q += split) {
        const int mm = mg * G + q;
        if (mm >= a.nmol) break;
        int *nl = s_nl + q * kMaxNeighbours, *off = s_off + q * (NS + 1);
        const int total = list_molecule(a.nb, L, iL, mm, NS, nl, off);
        if (chunk == 0) keep_list(a.nb, mm, NS, total, nl, off);
      }
      block_part_sync(32 * split);
    }
  }
  // each molecule takes half of every pair's energy and virial; a pair's
  // fixed-point force is the one on j
  const LjFix &lj = a.lj;
  LjSums s;
  bool took_f64 = false;
  double acc[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) acc[c] = 0.0;
  if (on && role < split) {
    // O-O Lennard-Jones: this warp's share of the buckets
    const int *off = own ? s_off + u * (NS + 1) : a.nb.off + (size_t)m * (NS + 1);
    const int *nl = own ? s_nl + u * kMaxNeighbours : a.nb.nbr + (size_t)m * kMaxNeighbours;
    int q = off[kSplit ? role * NS / split : 0];
    const int q1 = off[kSplit ? (role + 1) * NS / split : NS];
    int64_t LQ[3], xi[3];
    const int64_t *__restrict__ xp = a.xi + k;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      LQ[c] = fix_pos(L[c], lj.pos);
      xi[c] = xp[(size_t)(3 * m + c) * P];
    }
    PairF64 far;
    const int top = __double2hiint(lj.edge);   // the barostat may change the box
    const bool fixed =
        lj.on && __double2hiint(L[0]) < top && __double2hiint(L[1]) < top && __double2hiint(L[2]) < top;
    auto pair = [&](const int64_t (&xj)[3], int j) {
      if (fixed) {
        int64_t d[3];
        float h2 = 0.f;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          d[c] = fix_mic(xj[c] - xi[c], LQ[c]);
          const float h = (float)(int)(d[c] >> 32);
          h2 = fmaf(h, h, h2);
        }
        if (h2 >= lj.rpre2) return;
        if (lj_fix_pair<kDiag>(lj, d, s)) return;
      }
      pair_f64<kDiag>(a, L, iL, m, j, k, far);
    };
    // the next candidate's rows and the index after it are requested before
    // this candidate's arithmetic
    int j = q < q1 ? nl[q] : 0, jn = q + 1 < q1 ? nl[q + 1] : 0;
    int64_t xj[3], xn[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) xn[c] = xj[c] = xp[(size_t)(3 * j + c) * P];
#pragma unroll 1
    for (; q < q1; ++q) {
      const int ja = q + 2 < q1 ? nl[q + 2] : 0;
      if (q + 1 < q1) {
#pragma unroll
        for (int c = 0; c < 3; ++c) xn[c] = __ldg(xp + (size_t)(3 * jn + c) * P);
      }
      pair(xj, j);
      j = jn;
      jn = ja;
#pragma unroll
      for (int c = 0; c < 3; ++c) xj[c] = xn[c];
    }
    // the pairs taken in FP64
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      acc[c] = far.f[c];
      if (kDiag) acc[11 + c] = 0.5 * far.w3[c];
    }
    acc[9] = 0.5 * far.U;
    acc[10] = 0.5 * far.W;
    took_f64 = far.any;
  }
  if (!kSplit) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      acc[c] = fma(-lj.fs, fix_sum(s.f[c]), acc[c]);
      if (kDiag) acc[11 + c] = fma(0.5 * lj.w3, fix_sum(s.w[c]), acc[11 + c]);
    }
    acc[9] = fma(lj.us, fix_energy(s), acc[9]);
    acc[10] = fma(lj.ws, fix_sum(s.T), acc[10]);
  }
  if (on && (!kSplit || role >= split)) {
    Bonded b;
    bonded_f64<kDiag>(a, m, k, L, iL, b);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      acc[c] += b.fO[c];
      acc[3 + c] = b.fH[0][c];
      acc[6 + c] = b.fH[1][c];
      if (kDiag) acc[11 + c] += b.w3[c];
    }
    acc[9] += b.U;
    acc[10] += b.W;
  }
  auto store = [&](int comp, int mm, int kk, double v) {
    if (comp < 9)
      a.F[(size_t)(9 * mm + comp) * P + kk] = v;
    else if (comp == 9)
      a.Upart[(size_t)mm * P + kk] = v;
    else if (comp == 10)
      a.Wpart[(size_t)mm * P + kk] = v;
    else
      a.W3part[((size_t)mm * P + kk) * 3 + (comp - 11)] = v;
  };
  if (a.step_inc && blockIdx.x == 0 && threadIdx.x == 0) *a.step_inc += a.inc;
  if (!kSplit) {
    if (on)
#pragma unroll
      for (int c = 0; c < NC; ++c) store(c, m, k, acc[c]);
    return;
  }
  // partial sums joined in a fixed order, a component to a warp: the list's
  // fixed-point sums as integers (one conversion a component), its FP64 pairs
  // where a warp met one, the bonded warp's terms
  constexpr int NL = kDiag ? 8 : 5;    // f (3), T, y^3 (, w (3))
  constexpr int NF = kDiag ? 8 : 5;    // f (3), U, Tr Xi (, Xi_aa (3))
  __int128 *sI = reinterpret_cast<__int128 *>(s_off + ((G * (NS + 1) + 3) & ~3));   // [split][NL][32]
  double *sP = reinterpret_cast<double *>(sI + split * NL * 32);                    // [split][NF][32]
  double *sB = sP + split * NF * 32;                                                // [NC][32]
  __shared__ int s_f64[14];
  if (role < split) {
    const __int128 part[8] = {s.f[0], s.f[1], s.f[2], s.T, s.y3, s.w[0], s.w[1], s.w[2]};
#pragma unroll
    for (int c = 0; c < NL; ++c) sI[(role * NL + c) * 32 + lane] = part[c];
    const bool any = __any_sync(0xffffffffu, took_f64);
    if (lane == 0) s_f64[role] = any;
    if (any)
#pragma unroll
      for (int c = 0; c < NF; ++c) sP[(role * NF + c) * 32 + lane] = acc[c < 3 ? c : c + 6];
  } else {
#pragma unroll
    for (int c = 0; c < NC; ++c) sB[c * 32 + lane] = acc[c];
  }
  __syncthreads();
  for (int comp = warp; comp < NC; comp += split + 1) {   // the lanes keep their (molecule, bead)
    double sum = sB[comp * 32 + lane];
    if (comp < 3 || comp > 8) {   // the hydrogens' forces come from the bonded warp alone
      LjSums t;
      auto total = [&](int c) {
        __int128 v = 0;
        for (int w = 0; w < split; ++w) v += sI[(w * NL + c) * 32 + lane];
        return v;
      };
      double pair;
      if (comp < 3) {
        pair = -lj.fs * fix_sum(total(comp));
      } else if (comp == 9) {
        t.T = total(3);
        t.y3 = total(4);
        pair = lj.us * fix_energy(t);
      } else if (comp == 10) {
        pair = lj.ws * fix_sum(total(3));
      } else {
        pair = 0.5 * lj.w3 * fix_sum(total(comp - 6));
      }
      sum += pair;
      for (int w = 0; w < split; ++w)
        if (s_f64[w]) sum += sP[(w * NF + (comp < 3 ? comp : comp - 6)) * 32 + lane];
    }
    if (on) store(comp, m, k, sum);
  }
}

// The lists of a system's molecules, one warp each: on this step's skin test,
// or (force) always.  Small systems' force blocks do this themselves.
__global__ void __launch_bounds__(256) k_nbr_lists(NbrList a, int force) {
  if (!force && !skin_exceeded(a.blkmax, a.nblk_check, a.skin, blockDim.x)) return;
  const int NS = kLJWarps * a.groups, lane = threadIdx.x & 31;
  double L[3], iL[3];
  list_box(a, L, iL);
  for (int m = blockIdx.x * 8 + (threadIdx.x >> 5); m < a.nmol; m += gridDim.x * 8) {
    const int total = list_molecule(a, L, iL, m, NS, a.nbr + (size_t)m * kMaxNeighbours, a.off + (size_t)m * (NS + 1));
    if (total >= 0 && lane < 3) a.cref[3 * m + lane] = a.ccur[3 * m + lane];
  }
}

// Centroids of the oxygens from the positions (used when the positions were
// set from outside the step kernel: create, set_state), one lane group a row.
__global__ void k_centroids(int nmol, int P, const double *x, double *ccur) {
  const int W = row_lanes(P), l = threadIdx.x % W;
  const int r = (blockIdx.x * blockDim.x + threadIdx.x) / W;   // row 3 m + d
  double s = 0.0;
  if (r < 3 * nmol)
    for (int k = l; k < P; k += W) s += x[((size_t)9 * (r / 3) + r % 3) * P + k];
  s = group_sum(s, W);
  if (r < 3 * nmol && l == 0) ccur[r] = s / P;
}

// --- host launchers --------------------------------------------------------
int force_block_threads(int P) {
  // a whole number of bead groups per block, at least one warp
  int per = 128 / P;
  if (per < 1) per = 1;
  int t = per * P;
  if (t < 32) t = 32;
  return t;
}

int force_blocks(int n_groups, int P) {
  const int per = force_block_threads(P) / P;
  return (n_groups + per - 1) / per;
}

// Units of work of the water force (one molecule x 32 beads, or 32 / P molecules).
int water_units(int nmol, int P) {
  const int Bk = P < 32 ? P : 32, G = 32 / Bk;
  return (nmol + G - 1) / G * ((P + Bk - 1) / Bk);
}

// Warps that share a unit's neighbour list: each takes a range of consecutive
// buckets, [role NS / split, (role + 1) NS / split), equal in size where split
// divides NS (a multiple of 14) and one apart otherwise.
// 1, a warp takes whole units and makes no reduction, from eight units an SM on:
// us a step, split 1 against 4, 1024 units 68.1 against 66.4, 1200 73.2 against 73.8,
// 1400 84.0 against 85.9, 2048 106 against 117.  Below, warps are short of work and
// the list's chain is what counts: 4 against 7 at 432 units 33.1 against 39.2, at 160
// 25.0 against 23.9; 7 against 14 at 125 units (a block has its SM to itself) 19.9
// against 18.4.
static int water_split(int nmol, int P) {
  const int n = water_units(nmol, P);
  return n >= 1216 ? 1 : (n >= 192 ? 4 : (n > 152 ? 7 : 14));
}

// lane groups per warp of the water force kernel: the largest power of two
// <= min(8, 32 / min(P, 32))
int water_lane_groups(int P) {
  const int Bk = P < 32 ? P : 32;
  int g = 1;
  while (2 * g <= 8 && 2 * g * Bk <= 32) g *= 2;
  return g;
}

cudaError_t launch_force_harmonic(const ForceArgs &a, cudaStream_t s) {
  k_force_harmonic_f64<<<force_blocks(a.N, a.P), force_block_threads(a.P), 0, s>>>(a);
  return cudaGetLastError();
}

// Whether the list check is a kernel of its own (the one-warp units).
bool water_lists_apart(int nmol, int P) { return water_split(nmol, P) == 1; }

template <bool kDiag>
static void force_water(const ForceArgs &a, cudaStream_t s) {
  const int split = water_split(a.nmol, a.P), units = water_units(a.nmol, a.P);
  if (split == 1) {
    k_force_water_f64<kDiag, 0><<<(units + 3) / 4, 128, 0, s>>>(a, 1);
    return;
  }
  const int Bk = a.P < 32 ? a.P : 32, G = 32 / Bk, NS = kLJWarps * a.nb.groups;
  const size_t smem = (size_t)G * kMaxNeighbours * sizeof(int) + (((size_t)G * (NS + 1) + 3) & ~(size_t)3) * sizeof(int) +
                      ((size_t)split * (kDiag ? 8 : 5) * 3 + (kDiag ? 14 : 11)) * 32 * sizeof(double);
  if (split == 4)
    k_force_water_f64<kDiag, 2><<<units, 32 * (split + 1), smem, s>>>(a, split);
  else
    k_force_water_f64<kDiag, 1><<<units, 32 * (split + 1), smem, s>>>(a, split);
}

cudaError_t force_water_prepare() {   // a one-bead system's lists take more than 48 KB
  const int most = 160 * 1024;
  cudaError_t e = cudaFuncSetAttribute(k_force_water_f64<false, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_force_water_f64<false, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_force_water_f64<true, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_force_water_f64<true, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
  return e;
}

cudaError_t launch_force_water(const ForceArgs &a, cudaStream_t s) {
  if (a.W3part)
    force_water<true>(a, s);
  else
    force_water<false>(a, s);
  return cudaGetLastError();
}

// Wrapped fixed-point positions of the oxygens (the step kernels write them;
// this is for positions from outside).
__global__ void k_fix_positions(ForceArgs a, long long *xi) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= a.nmol * 3 * a.P) return;
  const int k = t % a.P, mc = t / a.P, c = mc % 3, m = mc / 3;
  double L[3], iL[3];
  list_box(a.nb, L, iL);
  const double x = a.x[(size_t)(9 * m + c) * a.P + k];
  xi[t] = fix_wrap(x, a.lj.pos, (float)x, (float)iL[c], fix_pos(L[c], a.lj.pos));
}

cudaError_t launch_fix_positions(const ForceArgs &a, long long *xi, cudaStream_t s) {
  const int n = a.nmol * 3 * a.P;
  k_fix_positions<<<(n + 255) / 256, 256, 0, s>>>(a, xi);
  return cudaGetLastError();
}

cudaError_t launch_nbr_lists(const NbrList &a, bool force, cudaStream_t s) {
  k_nbr_lists<<<std::min((a.nmol + 7) / 8, 304), 256, 0, s>>>(a, force ? 1 : 0);
  return cudaGetLastError();
}

cudaError_t launch_centroids(int nmol, int P, const double *x, double *ccur, cudaStream_t s) {
  const long long threads = (long long)3 * nmol * row_lanes(P);
  k_centroids<<<(unsigned)((threads + 127) / 128), 128, 0, s>>>(nmol, P, x, ccur);
  return cudaGetLastError();
}

}  // namespace pimd
