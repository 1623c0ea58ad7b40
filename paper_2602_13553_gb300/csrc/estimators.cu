// estimators.cu -- App. A outputs 1-10 reduced on the device, FP64.
//
// Pass 1 (k_est_f64): persistent blocks walk atom tiles of all P beads.
// Thread (atom al, mode k) forms q~_k = (M x)_k and adds
//   1/2 m |v~_k|^2            -> K^(k)   (output 1)
//   1/2 m w_n^2 lam_k |q~_k|^2 -> S^(k)   (output 2; sum_k S^(k) is the
//                                          ring's spring energy)
// and, as bead j = k, r^j . F^j and (r^j - r_c) . F^j (r_c = bead average),
// and its share of the force kernel's rows of U^(k) and Tr Xi^(k).  A thread
// keeps its (al, k) over all of its block's tiles, so every sum is one
// compensated chain (CSum) per thread; one row of partials per block.
// Pass 2 (k_est_final): blocks of eight columns sum the rows, 32 compensated
// chains per column and a fixed tree over them; the last block to finish
// assembles the outputs; a NaN/Inf sets the error word.  The order of every
// sum is fixed by the sizes alone.
//
// The FP64 pipe bounds pass 1 (two FMAs a clock and SM), so the tile is small
// where the system is (every SM gets atoms), the transform is folded (P / 2 + 1
// FMAs a mode), and the three components of a product share one compensated
// addition.  Pass 2 used to be one block with one serial chain per column:
// 65536 atoms x 32 beads 11.9 ms, 512 molecules x 64 beads 0.50 ms,
// 64 x 32 beads 51 us.
#include "common.cuh"

#include <algorithm>

namespace pimd {

__global__ void __launch_bounds__(256) k_est_f64(EstArgs a) {
  extern __shared__ double sm[];
  const int P = a.P, A = a.A, H = P >> 1;
  const int tileLen = A * 3 * P;
  double *sX = sm;
  double *sU = sX + tileLen;          // folded rows (normal modes) or v (Cartesian)
  double *sC = sU + tileLen;          // [A*3] centroids
  double *sB = sC + A * 3;            // [A*3] sum_k v^(k) (Cartesian)
  __shared__ CSum sR[4][256];
  __shared__ CSum sred[3][8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = (blockDim.x + 31) >> 5;
  const bool mine = (int)threadIdx.x < A * P;
  const int al = threadIdx.x / P, k = threadIdx.x - al * P;
  CSum kk{0.0, 0.0}, ss{0.0, 0.0}, uu{0.0, 0.0}, ww{0.0, 0.0};
  CSum rF{0.0, 0.0}, rcF{0.0, 0.0}, mv0{0.0, 0.0};
  // the force kernel's bead rows, dealt to the blocks like the atoms
  if (mine)
    for (int r = blockIdx.x * A + al; r < a.nblk_force; r += gridDim.x * A) {
      uu.add(a.Upart[(size_t)r * P + k]);
      ww.add(a.Wpart[(size_t)r * P + k]);
    }
  const double rsp = rsqrt((double)P);
  const double *__restrict__ Tf = a.mt.Tf;
  const int ntiles = (a.N + A - 1) / A;
  for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int tile0 = tile * A;
    const int na = min(A, a.N - tile0);
    const int len = na * 3 * P;
    const size_t base = (size_t)tile0 * 3 * P;
    const bool on = mine && al < na;
    double vv[3] = {0.0, 0.0, 0.0}, ff[3] = {0.0, 0.0, 0.0};
    if (on) {
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        vv[d] = a.v[base + (size_t)(al * 3 + d) * P + k];
        ff[d] = a.F[base + (size_t)(al * 3 + d) * P + k];
      }
    }
    __syncthreads();   // the previous tile is done with the shared rows
    for (int t = threadIdx.x; t < len; t += blockDim.x) {
      sX[t] = a.x[base + t];
      if (a.method == 1) sU[t] = a.v[base + t];
    }
    __syncthreads();
    double q[3] = {0.0, 0.0, 0.0};
    if (a.method == 0) {
      // rows folded as in the step kernel: u_j = x_j + x_{P-j}, u_{P-j} = x_j - x_{P-j}
      for (int t = threadIdx.x; t < na * 3 * (H + 1); t += blockDim.x) {
        const int r = t / (H + 1), j = t - r * (H + 1), pj = P - j;
        const double *xr = sX + r * P;
        double *ur = sU + r * P;
        if (j == 0 || pj == j) {
          ur[j] = xr[j];
        } else if (j < pj) {
          const double xa = xr[j], xb = xr[pj];
          ur[j] = xa + xb;
          ur[pj] = xa - xb;
        }
      }
      __syncthreads();
      if (on) {
        const bool even = k <= H;
        const int n = even ? H + 1 : P - H - 1;
        const double *u = sU + al * 3 * P + (even ? 0 : H + 1);
        const double *tf = Tf + k;
        for (int j = 0; j < n; ++j) {
          const double m = __ldg(tf + j * P);
          q[0] = fma(m, u[j], q[0]);
          q[1] = fma(m, u[P + j], q[1]);
          q[2] = fma(m, u[2 * P + j], q[2]);
        }
        if (k == 0)
#pragma unroll
          for (int d = 0; d < 3; ++d) sC[al * 3 + d] = q[d] * rsp;
      }
    } else {
      // row sums of x and v, one warp per row
      for (int r = warp; r < na * 3; r += nwarp) {
        double sx = 0.0, sv = 0.0;
        for (int j = lane; j < P; j += 32) {
          sx += sX[r * P + j];
          sv += sU[r * P + j];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          sx += __shfl_xor_sync(0xffffffffu, sx, o);
          sv += __shfl_xor_sync(0xffffffffu, sv, o);
        }
        if (lane == 0) {
          sC[r] = sx / P;
          sB[r] = sv;
        }
      }
    }
    __syncthreads();
    if (!on) continue;
    const double mm = __ldg(a.mass_mm + tile0 + al);
    const double v2s = vv[0] * vv[0] + vv[1] * vv[1] + vv[2] * vv[2];
    kk.add(0.5 * mm * __ldg(a.mt.mu + k) * v2s);   // fictitious mass m^(k)
    const double *xx = sX + al * 3 * P;
    if (a.method == 0) {
      ss.add(0.5 * mm * a.wn2 * __ldg(a.mt.lam + k) * (q[0] * q[0] + q[1] * q[1] + q[2] * q[2]));
      if (k == 0) mv0.add(mm * __ldg(a.mt.mu) * v2s);
    } else {
      // Cartesian bead form of output 2, and v~^(0) = sum_k v^(k) / sqrt(P)
      const int km = k == 0 ? P - 1 : k - 1, kp = k == P - 1 ? 0 : k + 1;
      double s2 = 0.0;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const double *xr = xx + d * P;
        const double dm = xr[k] - xr[km], dp = xr[k] - xr[kp];
        s2 += dm * dm + dp * dp;
      }
      ss.add(0.25 * mm * a.wn2 * s2);
      if (k == 0) {
        const double *b = sB + al * 3;
        mv0.add(mm * __ldg(a.mt.mu) * (b[0] * b[0] + b[1] * b[1] + b[2] * b[2]) / P);
      }
    }
    // bead j = k
    const double x0 = xx[k], x1 = xx[P + k], x2 = xx[2 * P + k];
    const double *c = sC + al * 3;
    rF.add(fma(x2, ff[2], fma(x1, ff[1], x0 * ff[0])));
    rcF.add(fma(x2 - c[2], ff[2], fma(x1 - c[1], ff[1], (x0 - c[0]) * ff[0])));
  }
  rF = warp_csum(rF);
  rcF = warp_csum(rcF);
  mv0 = warp_csum(mv0);
  if (lane == 0) {
    sred[0][warp] = rF;
    sred[1][warp] = rcF;
    sred[2][warp] = mv0;
  }
  sR[0][threadIdx.x] = kk;
  sR[1][threadIdx.x] = ss;
  sR[2][threadIdx.x] = uu;
  sR[3][threadIdx.x] = ww;
  __syncthreads();
  double *out = a.part + (size_t)blockIdx.x * est_columns(P);
  for (int t = threadIdx.x; t < 4 * P; t += blockDim.x) {
    const int w = t / P, kq = t - w * P;
    CSum s{0.0, 0.0};
    for (int b = 0; b < A; ++b) s.add(sR[w][b * P + kq]);
    out[t] = s.value();
  }
  if (threadIdx.x < 3) {
    CSum s{0.0, 0.0};
    for (int w = 0; w < nwarp; ++w) s.add(sred[threadIdx.x][w]);
    out[4 * P + threadIdx.x] = s.value();
  }
}

constexpr int kFinCols = 8;    // columns per block of pass 2
constexpr int kFinSegs = 32;   // row chains per column

__global__ void __launch_bounds__(kFinCols * kFinSegs) k_est_final(EstFinalArgs a) {
  __shared__ CSum sw[kFinCols][8];
  __shared__ double stot[4];
  __shared__ bool last;
  const int P = a.P, W = est_columns(P);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int c = threadIdx.x % kFinCols, seg = threadIdx.x / kFinCols;
  const int col = blockIdx.x * kFinCols + c;
  CSum s{0.0, 0.0};
  if (col < W)
    for (int r = seg; r < a.nblk_est; r += kFinSegs) s.add(a.part[(size_t)r * W + col]);
  // the four chains of a column in this warp, then the eight warps in order
#pragma unroll
  for (int o = 16; o >= kFinCols; o >>= 1) {
    CSum t{__shfl_down_sync(0xffffffffu, s.s, o), __shfl_down_sync(0xffffffffu, s.c, o)};
    s.add(t);
  }
  if (lane < kFinCols) sw[lane][warp] = s;
  __syncthreads();
  if (threadIdx.x < kFinCols && col < W) {
    CSum t{0.0, 0.0};
    for (int w = 0; w < 8; ++w) t.add(sw[threadIdx.x][w]);
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
    CSum t{0.0, 0.0};
    for (int k = lane; k < P; k += 32) t.add(__ldcg(a.tot + warp * P + k));
    t = warp_csum(t);
    if (lane == 0) stot[warp] = t.value();
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  const double Ktot = stot[0], Stot = stot[1], Utot = stot[2], Wtot = stot[3];
  const double rF = __ldcg(a.tot + 4 * P), rcF = __ldcg(a.tot + 4 * P + 1), mv0 = __ldcg(a.tot + 4 * P + 2);
  const double N = (double)a.N, Pd = (double)P, kT = a.kT;
  const double V = a.dbox ? a.dbox[0] * a.dbox[1] * a.dbox[2] : a.volume;
  const double spring = 2.0 * Stot;   // sum_k sum_i m w_n^2 |r^k - r^(k+1)|^2
  double *g = o + 3 * P;
  g[0] = Ktot + Stot + Utot;                                    // H
  g[1] = 1.5 * Pd * N * kT - 0.5 * spring / Pd;                 // K_PR
  g[2] = -rF / (2.0 * Pd);                                      // K_VR
  g[3] = 1.5 * N * kT - rcF / (2.0 * Pd);                       // K_CV
  if (V > 0.0) {
    g[4] = (3.0 * Pd * N * kT - spring / Pd + Wtot / Pd) / (3.0 * V);  // P_PR
    g[5] = (2.0 * Ktot + Wtot) / (3.0 * V);                            // P_MD
    g[6] = (mv0 - rcF + Wtot) / (3.0 * Pd * V);                        // P_CV
  } else {
    const double nan = __longlong_as_double(0x7ff8000000000000ll);
    g[4] = g[5] = g[6] = nan;
  }
  g[7] = 2.0 * Ktot / (3.0 * N * Pd * a.kB);                   // T_ring
  g[8] = V;
  g[9] = Wtot;
  bool finite = isfinite(g[0]) && isfinite(g[1]) && isfinite(g[2]) && isfinite(g[3]);
  if (!finite) atomicOr(a.err, kErrNonFinite);
}

size_t est_smem_bytes(int A, int P) { return (size_t)(2 * A * 3 * P + 6 * A) * sizeof(double); }

// Rows of partials: one per block, four blocks per SM at most.
int est_rows(int N, int A) { return std::min((N + A - 1) / A, 608); }

cudaError_t launch_est(const EstArgs &a, int threads, cudaStream_t s) {
  k_est_f64<<<est_rows(a.N, a.A), threads, est_smem_bytes(a.A, a.P), s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_est_final(const EstFinalArgs &a, cudaStream_t s) {
  k_est_final<<<(est_columns(a.P) + kFinCols - 1) / kFinCols, kFinCols * kFinSegs, 0, s>>>(a);
  return cudaGetLastError();
}

}  // namespace pimd
