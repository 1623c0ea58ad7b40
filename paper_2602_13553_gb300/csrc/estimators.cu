// estimators.cu -- App. A outputs 1-10 reduced on the device, FP64.
//
// Pass 1 (k_est_f64): persistent blocks walk atom tiles of all P beads.
// Thread (atom al, mode k) forms q~_k = (M x)_k and adds
//   1/2 m |v~_k|^2            -> K^(k)   (output 1)
//   1/2 m w_n^2 lam_k |q~_k|^2 -> S^(k)   (output 2; sum_k S^(k) is the
//                                          ring's spring energy)
// and, as bead j = k, r^j . F^j and (r^j - r_c) . F^j (r_c = bead average),
// and its share of the force kernel's rows of U^(k) and Tr Xi^(k).  A thread
// keeps its (al, k) over all of its block's tiles, so every sum is one chain
// per thread; one row of partials per block.
// Pass 2 (k_est_final): blocks of eight columns sum the rows, 32 chains per
// column and a fixed tree over them; the last block to finish assembles the
// outputs, one per lane; a NaN/Inf sets the error word.  The order of every sum
// is fixed by the sizes alone.
//
// What bounds both is the FP64 pipe (one warp instruction in 64 clocks per SM
// partition), and in small systems the length of its dependent chains.  So the
// transform runs in fixed point as in the step kernel, every sum is a 128-bit
// integer (wide.cuh: ~30 integer instructions a term where a compensated FP64
// addition takes 450 clocks), factors common to a column are multiplied in once
// at its end, and no two divisions follow each other but those of one output:
// 20 FP64 instructions an (atom, mode) are left, of 109.  Pass 1 / pass 2, with
// compensated FP64 sums before and now: 65536 atoms x 32 beads 581 / 21 -> 189 /
// 15 us; 512 molecules x 64 beads 77 / 19 -> 26 / 11; 64 x 32 beads 16 / 16 ->
// 8.8 / 9.2.  The tile is small where the system is, so every SM gets atoms.
#include "common.cuh"
#include "fixed.cuh"
#include "wide.cuh"

#include <algorithm>

namespace pimd {

template <bool kCart>
__global__ void __launch_bounds__(256) k_est_f64(EstArgs a) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const int P = a.P, A = a.A, H = P >> 1, AP = A * P, np = fix_pairs(P), rs = 4 * np;
  // normal modes: folded limbs, fixed-point rows; Cartesian: x and v
  int4 *uX = reinterpret_cast<int4 *>(smraw);                        // [3A][rs / 2]
  long long *rX = reinterpret_cast<long long *>(uX + 3 * A * (rs >> 1));   // [3A][P]
  double *sX = reinterpret_cast<double *>(smraw);                    // [3A][P]
  double *sV = sX + 3 * AP;                                          // [3A][P]
  WideSum *sR = reinterpret_cast<WideSum *>(smraw);                  // [4][AP], after the tiles
  __shared__ double sC[3 * 256];   // centroids
  __shared__ double sB[3 * 256];   // sum_k v^(k) (Cartesian)
  __shared__ int sE[3 * 256];      // largest exponents of the rows
  __shared__ WideSum sred[3][8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = (blockDim.x + 31) >> 5;
  const bool mine = (int)threadIdx.x < AP;
  const int al = threadIdx.x / P, k = threadIdx.x - al * P;
  WideSum kk, ss, rF, rcF, mv0;
  kk.clear();
  ss.clear();
  rF.clear();
  rcF.clear();
  mv0.clear();
  const double rsp = a.mt.rsp;
  const int pj = k == 0 ? 0 : P - k;
  const bool even = k <= H;
  const int em = a.mt.fem;
  const int4 *__restrict__ tf = a.mt.fTf + (mine ? k : 0);
  if (!kCart)
    for (int t = threadIdx.x; t < 3 * A; t += blockDim.x) sE[t] = kFixMinE;
  const int ntiles = (a.N + A - 1) / A;
  for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int tile0 = tile * A;
    const int na = min(A, a.N - tile0);
    const bool on = mine && al < na;
    double x[3] = {0.0, 0.0, 0.0}, v[3] = {0.0, 0.0, 0.0}, f[3] = {0.0, 0.0, 0.0};
    double mm = 0.0;
    if (on) {
      const size_t g = ((size_t)(tile0 + al) * 3) * P + k;
#pragma unroll
      for (int d = 0; d < 3; ++d) x[d] = a.x[g + (size_t)d * P];
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        v[d] = a.v[g + (size_t)d * P];
        f[d] = a.F[g + (size_t)d * P];
      }
      mm = __ldg(a.mass_mm + tile0 + al);
    }
    __syncthreads();   // the previous tile is done with the shared rows
    if (!kCart) {
      if (on)
#pragma unroll
        for (int d = 0; d < 3; ++d) atomicMax(sE + al * 3 + d, exp_field(x[d]));
      __syncthreads();
      int E[3];
      long long X[3];
      if (on)
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          E[d] = sE[al * 3 + d];
          rX[(al * 3 + d) * P + k] = X[d] = to_fixed(x[d], E[d]);
        }
      __syncthreads();
      if (on)   // folded as in the step: u_j = x_j + x_{P-j}, u_{P-j} = x_{P-j} - x_j
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          const int r = al * 3 + d;
          const long long o = pj != k ? rX[r * P + pj] : 0;
          reinterpret_cast<int2 *>(uX)[r * rs + (even ? k : 2 * np + k - H - 1)] = fix_limbs(even ? X[d] + o : o - X[d]);
          if (k == 0) sE[r] = kFixMinE;   // for the next tile
        }
      __syncthreads();
      if (on) {
        const int4 *u = uX + al * 3 * (rs >> 1) + (even ? 0 : np);
        FixSum s[3];
        for (int p = 0; p < np; ++p) {
          const int4 m = __ldg(tf + p * P);
#pragma unroll
          for (int d = 0; d < 3; ++d) s[d].add2(u[d * (rs >> 1) + p], m);
        }
        double q2 = 0.0;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          const double q = from_fixed(s[d].value(), E[d], em);
          q2 = fma(q, q, q2);
          if (k == 0) sC[al * 3 + d] = q * rsp;
        }
        ss.add(mm * q2);
      }
      __syncthreads();
    } else {
      if (on)
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          sX[(al * 3 + d) * P + k] = x[d];
          sV[(al * 3 + d) * P + k] = v[d];
        }
      __syncthreads();
      // row sums of x and v, one warp per row
      for (int r = warp; r < na * 3; r += nwarp) {
        double sx = 0.0, sv = 0.0;
        for (int j = lane; j < P; j += 32) {
          sx += sX[r * P + j];
          sv += sV[r * P + j];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          sx += __shfl_xor_sync(0xffffffffu, sx, o);
          sv += __shfl_xor_sync(0xffffffffu, sv, o);
        }
        if (lane == 0) {
          sC[r] = sx;
          sB[r] = sv;
        }
      }
      __syncthreads();
      for (int t = threadIdx.x; t < na * 3; t += blockDim.x) sC[t] /= P;
      if (on) {
        // Cartesian bead form of output 2, and v~^(0) = sum_k v^(k) / sqrt(P)
        const double *xx = sX + al * 3 * P;
        const int km = k == 0 ? P - 1 : k - 1, kp = k == P - 1 ? 0 : k + 1;
        double s2 = 0.0;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          const double dm = x[d] - xx[d * P + km], dp = x[d] - xx[d * P + kp];
          s2 = fma(dp, dp, fma(dm, dm, s2));
        }
        ss.add(mm * s2);
        if (k == 0) {
          const double *b = sB + al * 3;
          mv0.add(mm * (b[0] * b[0] + b[1] * b[1] + b[2] * b[2]));
        }
      }
      __syncthreads();
    }
    if (!on) continue;
    kk.add(mm * fma(v[2], v[2], fma(v[1], v[1], v[0] * v[0])));
    // bead j = k
    rF.add(fma(x[2], f[2], fma(x[1], f[1], x[0] * f[0])));
    const double *c = sC + al * 3;
    rcF.add(fma(x[2] - c[2], f[2], fma(x[1] - c[1], f[1], (x[0] - c[0]) * f[0])));
  }
  rF = warp_wide(rF);
  rcF = warp_wide(rcF);
  if (kCart) mv0 = warp_wide(mv0);
  if (lane == 0) {
    sred[0][warp] = rF;
    sred[1][warp] = rcF;
    sred[2][warp] = mv0;
  }
  // the force kernel's bead rows, dealt to the blocks like the atoms
  WideSum uu, ww;
  uu.clear();
  ww.clear();
  if (mine)
    for (int r = blockIdx.x * A + al; r < a.nblk_force; r += gridDim.x * A) {
      uu.add(a.Upart[(size_t)r * P + k]);
      ww.add(a.Wpart[(size_t)r * P + k]);
    }
  // the A chains of a mode (bead), halved until one is left
  __syncthreads();
  WideSum *mineR = sR + threadIdx.x;
  if (mine) {
    mineR[0] = kk;
    mineR[AP] = ss;
    mineR[2 * AP] = uu;
    mineR[3 * AP] = ww;
  }
  for (int n = A; n > 1;) {
    const int half = (n + 1) >> 1;
    __syncthreads();
    if (mine && al + half < n) {
#pragma unroll
      for (int w = 0; w < 4; ++w) mineR[w * AP].add(mineR[w * AP + half * P]);
    }
    n = half;
  }
  __syncthreads();
  double *out = a.part + (size_t)blockIdx.x * est_columns(P);
  for (int t = threadIdx.x; t < 4 * P; t += blockDim.x) {
    const int w = t / P, kq = t - w * P;
    double s = sR[w * AP + kq].value();
    if (w == 0) s *= 0.5 * __ldg(a.mt.mu + kq);   // fictitious mass m^(k)
    if (w == 1) s *= kCart ? 0.25 * a.wn2 : 0.5 * a.wn2 * __ldg(a.mt.lam + kq);
    out[t] = s;
    // 2 K of the centroid mode
    if (!kCart && t == 0) out[4 * P + 2] = 2.0 * s;
  }
  if ((int)threadIdx.x < (kCart ? 3 : 2)) {
    WideSum s = sred[threadIdx.x][0];
    for (int w = 1; w < nwarp; ++w) s.add(sred[threadIdx.x][w]);
    out[4 * P + threadIdx.x] = s.value() * (threadIdx.x == 2 ? __ldg(a.mt.mu) / P : 1.0);
  }
}

constexpr int kFinCols = 8;    // columns per block of pass 2
constexpr int kFinSegs = 32;   // row chains per column

__global__ void __launch_bounds__(kFinCols * kFinSegs) k_est_final(EstFinalArgs a) {
  __shared__ WideSum sw[kFinCols][8];
  __shared__ double stot[4];
  __shared__ bool last;
  const int P = a.P, W = est_columns(P);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int c = threadIdx.x % kFinCols, seg = threadIdx.x / kFinCols;
  const int col = blockIdx.x * kFinCols + c;
  WideSum s;
  s.clear();
  if (col < W) {
#pragma unroll 4
    for (int r = seg; r < a.nblk_est; r += kFinSegs) s.add(a.part[(size_t)r * W + col]);
  }
  // the four chains of a column in this warp, then the eight warps in order
#pragma unroll
  for (int o = 16; o >= kFinCols; o >>= 1) s.add(s.shfl_down(o));
  if (lane < kFinCols) sw[lane][warp] = s;
  __syncthreads();
  if (threadIdx.x < kFinCols && col < W) {
    WideSum t = sw[threadIdx.x][0];
#pragma unroll
    for (int w = 1; w < 8; ++w) t.add(sw[threadIdx.x][w]);
    a.tot[col] = t.value();
    __threadfence();
  }
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(a.count, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  if (threadIdx.x == 0) *a.count = 0;   // for the next call on this handle
  double *o = a.out;
  for (int t = threadIdx.x; t < 3 * P; t += blockDim.x) o[t] = __ldcg(a.tot + t);
  if (warp < 4) {   // sums over the modes (beads) of K, S, U and Tr Xi, one warp each
    WideSum t;
    t.clear();
    for (int k = lane; k < P; k += 32) t.add(__ldcg(a.tot + warp * P + k));
    t = warp_wide(t);
    if (lane == 0) stot[warp] = t.value();
  }
  __syncthreads();
  if (threadIdx.x >= 10) return;
  // one output per lane, ((a + b) / c + d) / e: two divisions deep, not ten in a row
  const double Ktot = stot[0], Stot = stot[1], Utot = stot[2], Wtot = stot[3];
  const double rF = __ldcg(a.tot + 4 * P), rcF = __ldcg(a.tot + 4 * P + 1), mv0 = __ldcg(a.tot + 4 * P + 2);
  const double Pd = (double)P, NkT = (double)a.N * a.kT;
  const double V = a.dbox ? a.dbox[0] * a.dbox[1] * a.dbox[2] : a.volume;
  const double spring = 2.0 * Stot;   // sum_k sum_i m w_n^2 |r^k - r^(k+1)|^2
  double num = 0.0, den = Pd, add = 0.0, den2 = 1.0;
  switch (threadIdx.x) {
    case 0: add = Ktot + Stot + Utot; break;                                     // H
    case 1: num = -0.5 * spring, add = 1.5 * Pd * NkT; break;                    // K_PR
    case 2: num = -0.5 * rF; break;                                              // K_VR
    case 3: num = -0.5 * rcF, add = 1.5 * NkT; break;                            // K_CV
    case 4: num = Wtot - spring, add = 3.0 * Pd * NkT, den2 = 3.0 * V; break;    // P_PR
    case 5: add = 2.0 * Ktot + Wtot, den2 = 3.0 * V; break;                      // P_MD
    case 6: num = mv0 - rcF + Wtot, den2 = 3.0 * V; break;                       // P_CV
    case 7: num = 2.0 * Ktot, den2 = 3.0 * (double)a.N * a.kB; break;            // T_ring
    case 8: add = V; break;
    default: add = Wtot; break;
  }
  double g = (num / den + add) / den2;
  if (threadIdx.x >= 4 && threadIdx.x < 7 && !(V > 0.0)) g = __longlong_as_double(0x7ff8000000000000ll);
  o[3 * P + threadIdx.x] = g;
  if (threadIdx.x < 4 && !isfinite(g)) atomicOr(a.err, kErrNonFinite);
}

size_t est_smem_bytes(int A, int P, bool cart) {
  const size_t rows = cart ? (size_t)2 * 3 * A * P * sizeof(double)
                           : (size_t)3 * A * (2 * fix_pairs(P) * sizeof(int4) + P * sizeof(long long));
  return std::max(rows, (size_t)4 * A * P * sizeof(WideSum));
}

// Rows of partials: one per block, four blocks per SM at most.
int est_rows(int N, int A) { return std::min((N + A - 1) / A, 608); }

cudaError_t launch_est(const EstArgs &a, int threads, cudaStream_t s) {
  const int rows = est_rows(a.N, a.A);
  if (a.method == 1)
    k_est_f64<true><<<rows, threads, est_smem_bytes(a.A, a.P, true), s>>>(a);
  else
    k_est_f64<false><<<rows, threads, est_smem_bytes(a.A, a.P, false), s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_est_final(const EstFinalArgs &a, cudaStream_t s) {
  k_est_final<<<(est_columns(a.P) + kFinCols - 1) / kFinCols, kFinCols * kFinSegs, 0, s>>>(a);
  return cudaGetLastError();
}

}  // namespace pimd
