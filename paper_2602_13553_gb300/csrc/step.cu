// step.cu -- the fused normal-mode integrator step of the PIMD method
// (Sec. IV.A; App. B normal modes; App. D PILE_L), FP64.
//
// One thread block owns a tile of A atoms with all P beads of every one of
// them on chip, so the three normal-mode transforms of a step (forces,
// positions forward; positions back) never leave the SM: the inter-bead
// communication of the paper's MPI design becomes shared-memory traffic.  Per
// step and atom tile the kernel reads x, v~, F once and writes x, v~ once,
// coalesced (every atom's P beads are contiguous per component).
//
// Thread (component c, atom a, mode k) forms
//   F~_k = sum_j M[k][j] F_j and q~_k = sum_j M[k][j] x_j        (Eq. A1)
// applies B / A / O / A (BAOAB) or the pending B O of the previous step then
// O B A (OBABO) in registers, and stores v~; after a barrier, thread
// (c, a, bead j) forms x_j = sum_k M[k][j] q~_k (Eq. A3).
// For water-like systems the same kernel also measures, per oxygen, the
// centroid drift since the last neighbour-list build and the bead spread.
#include "common.cuh"
#include "fixed.cuh"

#include <algorithm>

namespace pimd {

__device__ __forceinline__ void rotate(double &q, double &v, double c, double s_over_w, double w_s) {
  // exact flow of a free-ring-polymer mode for time tA:
  //   q' = cos q + sin/w v,  v' = -w sin q + cos v   (k = 0: q' = q + tA v)
  const double qn = fma(c, q, s_over_w * v);
  const double vn = fma(-w_s, q, c * v);
  q = qn;
  v = vn;
}

// Centroid mode under the barostat for time tA at v_W (App. E):
//   q~0 <- e^a q~0 + (e^a - e^-a) / (2 v_W) v~0,  v~0 <- e^-a v~0,  a = tA v_W
// with the three factors as the barostat's kick left them.
__device__ __forceinline__ void baro_drift(double &q, double &v, const double *f) {
  q = f[0] * q + f[2] * v;
  v = f[1] * v;
}

__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_down_sync(0xffffffffu, v, o));
  return v;
}

// The fused step.  What bounds it is the FP64 pipe (one warp instruction in 64
// clocks per SM partition), so everything that can be is taken off it:
//  * the transforms run in 64-bit fixed point on the integer pipe (fixed.cuh),
//    folded by the parity of the rows of M (Eq. A1) under j -> P - j: modes
//    k <= H = floor(P/2) (constant, cosine and alternating rows) are even, the
//    sine rows k > H odd, so u_j = x_j + x_{P-j} and u_{P-j} = x_{P-j} - x_j
//    leave each output a sum over one half of the row (tables fTf, fTi), and the
//    inverse pair x_j, x_{P-j} = C_j +- S_j an even-mode and an odd-mode sum;
//  * A O A is one linear map of (q~, v~, eta) per mode (table map6);
//  * one Philox draw's Box-Muller work is dealt to the three threads of an
//    (atom, mode): the radius of the x, y pair, its angle, and all of z;
//  * scalings are exponent additions; the skin test and the force kernel's
//    wrapped fixed-point positions of the oxygens come from the integers.
// Threads are component-major (c = threadIdx.x / S, S whole warps), so a warp
// has one component and its Box-Muller share does not diverge.
//
// In a harmonic well (kHarm) F = -k x, so F~ = -k q~ and the forces are neither
// read nor transformed; the force kernel runs once, after a call's last step.
//
// kPhase 0: the whole step.  1, 2: a step in two launches around the barostat's
// OBABO kick (velocities only; then B(h/2), A(h) and the positions).  3: the
// closing B(h/2) (OBABO: and O(h/2)) of a call's last step.
//
// Measured, us a launch, with FP64 transforms and noise and the forces read
// against now: 65536 oscillators x 32 beads 1724 (and 61 of the force kernel) /
// 259 (FP64 instructions 160, issue 186 of it), 512 molecules x 64 beads 121 / 28,
// 64 x 32 14.4 / 7.6.
template <int kPhase, bool kObabo, bool kHarm>
__global__ void __launch_bounds__(384) k_step_f64(StepArgs a) {
  constexpr bool kX = kPhase == 0 || kPhase == 2;   // positions move
  constexpr bool kQ = kX || kHarm;                  // q~ is formed
  extern __shared__ __align__(16) unsigned char smraw[];
  const int P = a.P, H = P >> 1, A = a.A, AP = A * P, np = fix_pairs(P), rs = 4 * np;
  const int S = blockDim.x / 3;
  const int c = threadIdx.x / S, u = threadIdx.x - c * S;
  const int al = u / P, k = u - al * P;
  const int tile0 = blockIdx.x * A;
  const int na = min(A, a.N - tile0);
  const bool on = u < na * P;
  const int i = tile0 + al, row = c * A + min(al, A - 1);   // padding threads stay inside the rows
  const size_t g = ((size_t)i * 3 + c) * P + k;
  int4 *uX = reinterpret_cast<int4 *>(smraw);                 // folded limbs, rs / 2 per row
  int4 *uF = uX + 3 * A * (rs >> 1);
  long long *rX = reinterpret_cast<long long *>(uF + 3 * A * (rs >> 1));   // [3][AP]
  long long *rF = rX + 3 * AP;
  long long *sC = rF + 3 * AP;                                // [3A] centroids, fixed point
  uint64_t *sR = reinterpret_cast<uint64_t *>(sC + 3 * A);    // [2][AP] Box-Muller radius of x, y
  int64_t *sCs = reinterpret_cast<int64_t *>(sR + 2 * AP);    // [2][AP] cosine of their angle
  int *sE = reinterpret_cast<int *>(sCs + 2 * AP);            // [3][3A] largest exponents of x, F, q~
  float *sD = reinterpret_cast<float *>(sE + 9 * A);          // [3][AP] bead deviations
  __shared__ float sred[2][12];
  const bool needF = !kHarm && (kPhase != 1 || !a.first);
  double x = 0.0, f = 0.0, v = 0.0;
  if (on) {
    if (kQ) x = a.x[g];
    if (needF) f = a.F[g];
    v = a.v[g];
  }
  for (int t = threadIdx.x; t < 9 * A; t += blockDim.x) sE[t] = kFixMinE;
  const uint64_t step = (uint64_t)(*a.step + a.step_off);
  // the noise does not wait for the loads above: stream O1 of this step, O2 of
  // the previous one
  const bool d1 = a.thermo && (kPhase == 0 || kPhase == 1);
  const bool d2 = kObabo && a.thermo && kPhase != 2 && (kPhase == 3 || !a.first);
  double eta[2] = {0.0, 0.0};
  uint64_t part[2] = {0, 0};   // this thread's share: radius (c = 0) or sine (c = 1)
  auto draw = [&](int d, uint32_t stream, uint64_t st) {
    const uint4 w = noise_words(a.seed, (uint32_t)i, (uint32_t)k, stream, st);
    if (c == 0) {
      sR[d * AP + u] = part[d] = bm_radius_fix(w.x);
    } else {
      int64_t sn, cs;
      bm_angle_fix(c == 1 ? w.y : w.w, sn, cs);
      if (c == 1) {
        part[d] = (uint64_t)sn;
        sCs[d * AP + u] = cs;
      } else {
        eta[d] = bm_deviate(bm_radius_fix(w.z), cs);
      }
    }
  };
  if (on && d1) draw(0, kStreamO1, step);
  if (on && d2) draw(1, kStreamO2, step - 1);
  __syncthreads();
  if (on) {
    if (kQ) atomicMax(sE + row, exp_field(x));
    if (needF) atomicMax(sE + 3 * A + row, exp_field(f));
    if (c < 2) {   // e_x = r cos, e_y = r sin
#pragma unroll
      for (int d = 0; d < 2; ++d)
        if (d ? d2 : d1)
          eta[d] = c == 0 ? bm_deviate(part[d], sCs[d * AP + u]) : bm_deviate(sR[d * AP + u], (int64_t)part[d]);
    }
  }
  __syncthreads();
  const int Ex = sE[row], Ef = sE[3 * A + row];
  const int pj = k == 0 ? 0 : P - k;
  const bool even = k <= H;
  const int fold = row * rs + (even ? k : 2 * np + k - H - 1);   // this element's folded place
  const int half_row = row * (rs >> 1) + (even ? 0 : np);        // the terms of mode (bead) k
  long long X = 0, F = 0;
  if (on) {
    if (kQ) rX[c * AP + u] = X = to_fixed(x, Ex);
    if (needF) rF[c * AP + u] = F = to_fixed(f, Ef);
  }
  __syncthreads();
  if (on) {
    if (kQ) {
      const long long o = pj != k ? rX[c * AP + u - k + pj] : 0;
      reinterpret_cast<int2 *>(uX)[fold] = fix_limbs(even ? X + o : o - X);
    }
    if (needF) {
      const long long o = pj != k ? rF[c * AP + u - k + pj] : 0;
      reinterpret_cast<int2 *>(uF)[fold] = fix_limbs(even ? F + o : o - F);
    }
  }
  __syncthreads();
  const int em = a.mt.fem;
  const int4 *__restrict__ tf = a.mt.fTf + k;
  double q = 0.0;
  if (on) {
    FixSum sx, sf;
    if (kHarm) {
#pragma unroll 3
      for (int p = 0; p < np; ++p) sx.add2(uX[half_row + p], __ldg(tf + p * P));
      q = from_fixed(sx.value(), Ex, em);
    } else if (kX && needF) {
#pragma unroll 3
      for (int p = 0; p < np; ++p) {
        const int4 m = __ldg(tf + p * P);
        sx.add2(uX[half_row + p], m);
        sf.add2(uF[half_row + p], m);
      }
      q = from_fixed(sx.value(), Ex, em);
    } else if (needF) {
#pragma unroll 3
      for (int p = 0; p < np; ++p) sf.add2(uF[half_row + p], __ldg(tf + p * P));
    }
    f = kHarm ? -__ldg(a.kspring + i) * q : (needF ? from_fixed(sf.value(), Ef, em) : 0.0);
    if (!a.mu_one) f *= __ldg(a.mt.imu + k);   // 1 / m^(k) = imu_k / (m mvv2e)
    if (k == 0 && a.fix_u) v -= a.fix_u[c];    // the previous step's fixcom
    const double km = __ldg(a.kmm + i);        // this kick's time / (m mvv2e)
    const double sg = __ldg(a.sigv + i);
    if (!kObabo) {
      // B(h/2) of this step, merged with the final B(h/2) of the previous one
      v = fma(km, f, v);
      if (kPhase != 3) {
        const double n = sg * eta[0];
        if (k == 0 && a.baro) {   // the centroid rides on the barostat
          baro_drift(q, v, a.baro + kBaroA1 + 3 * c);
          if (a.thermo) v = fma(__ldg(a.mt.c1), v, __ldg(a.mt.c2) * n);
          baro_drift(q, v, a.baro + kBaroA2 + 3 * c);
        } else {
          // A(h/2) O(h) A(h/2): (q~, v~) <- linear map of (q~, v~, sigma eta)
          const double *__restrict__ m6 = a.mt.map6 + k;
          const double qn = fma(__ldg(m6 + 2 * P), n, fma(__ldg(m6 + P), v, __ldg(m6) * q));
          v = fma(__ldg(m6 + 5 * P), n, fma(__ldg(m6 + 4 * P), v, __ldg(m6 + 3 * P) * q));
          q = qn;
        }
      }
    } else {
      const double c1 = __ldg(a.mt.c1 + k), c2s = __ldg(a.mt.c2 + k) * sg;
      if (kPhase != 2) {
        if (kPhase == 3 || !a.first) {
          // the previous step's closing B(h/2) O(h/2)
          v = fma(km, f, v);
          if (a.thermo) v = fma(c1, v, c2s * eta[1]);
        }
        if (kPhase != 3 && a.thermo) v = fma(c1, v, c2s * eta[0]);
      }
      if (kX) {
        v = fma(km, f, v);
        if (k == 0 && a.baro)   // A(h) of the centroid under the barostat
          baro_drift(q, v, a.baro + kBaroA1 + 3 * c);
        else
          rotate(q, v, __ldg(a.mt.cA + k), __ldg(a.mt.sA + k), __ldg(a.mt.wsA + k));
      }
    }
    a.v[g] = v;
    if (kX) atomicMax(sE + 6 * A + row, exp_field(q));
  }
  if (!kX) return;
  __syncthreads();
  const int Eq = sE[6 * A + row];
  const int sh = Eq - 1022 + em - kFixBits;   // x_j = S_j 2^sh below
  const bool oxy = a.blkmax && on && i % 3 == 0;
  double cen = 0.0;
  if (on) {
    reinterpret_cast<int2 *>(uX)[fold] = fix_limbs(to_fixed(q, Eq));
    if (oxy && k == 0) {   // centroid c = q~_0 / sqrt(P), also in units of 2^sh
      cen = q * a.mt.rsp;
      sC[row] = Eq > kFixMaxE ? 0
                              : __double2ll_rn(__hiloint2double(__double2hiint(cen) - (sh << 20), __double2loint(cen)));
      if (cen == 0.0) sC[row] = 0;
    }
  }
  __syncthreads();
  // inverse, first half: C_j (bead j <= H, even modes) or S_{P-j} (bead
  // j > H, odd modes)
  if (on) {
    const int4 *__restrict__ ti = a.mt.fTi + k;
    FixSum s;
#pragma unroll 3
    for (int p = 0; p < np; ++p) s.add2(uX[half_row + p], __ldg(ti + p * P));
    rX[c * AP + u] = X = s.value();
  }
  __syncthreads();
  // second half: x_j = C_j + S_j (j <= H), x_{P-j} = C_j - S_j
  float dev = 0.f;
  if (on) {
    const long long o = rX[c * AP + u - k + pj];
    const long long Sj = even ? (pj > H ? X + o : X) : o - X;
    const double xn = from_fixed(Sj, Eq, em);
    a.x[g] = xn;
    if (oxy) {
      const float sc = sh < -126 ? 0.f : (sh > 127 ? __int_as_float(0x7f800000) : __int_as_float((sh + 127) << 23));
      const double Lc = a.dbox ? a.dbox[c] : a.box[c], iLc = a.dbox ? a.dbox[3 + c] : a.invbox[c];
      a.xi[((size_t)i + c) * P + k] = fix_wrap(xn, a.pos, (float)Sj * sc, (float)iLc, fix_pos(Lc, a.pos));   // row 3 (i / 3) + c
      dev = Eq > kFixMaxE ? __int_as_float(0x7f800000) : (float)(Sj - sC[row]) * sc;
      sD[c * AP + u] = dev;
    }
  }
  if (!a.blkmax) return;
  // Neighbour-list skin check for the oxygens of this tile: the centroid's
  // drift since the last build and the bead spread, squared and reduced in
  // FP32 (a relative margin keeps the reported bound conservative).  Tiles
  // without an oxygen report zero at once.
  if ((tile0 + 2) / 3 * 3 >= tile0 + na) {
    if (threadIdx.x < 2) a.blkmax[2 * blockIdx.x + threadIdx.x] = 0.0;
    return;
  }
  float *sG = reinterpret_cast<float *>(sE);   // [3][A] squared drifts (the exponents are done with)
  if (oxy && k == 0) {
    const int m = i / 3;
    const float d = (float)(cen - a.cref[3 * m + c]);
    a.ccur[3 * m + c] = cen;
    sG[row] = d * d;
  }
  __syncthreads();
  float vdisp = 0.f, vdev = 0.f;
  if (c == 0 && oxy) {
    const float e1 = sD[AP + u], e2 = sD[2 * AP + u];
    vdev = dev * dev + e1 * e1 + e2 * e2;
    if (k == 0) vdisp = sG[al] + sG[A + al] + sG[2 * A + al];
    // NaN positions force a rebuild (and fail later at a synchronising call)
    if (vdisp != vdisp) vdisp = __int_as_float(0x7f800000);
    if (vdev != vdev) vdev = __int_as_float(0x7f800000);
  }
  if (c == 0) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      vdisp = fmaxf(vdisp, __shfl_down_sync(0xffffffffu, vdisp, o));
      vdev = fmaxf(vdev, __shfl_down_sync(0xffffffffu, vdev, o));
    }
    if ((threadIdx.x & 31) == 0) {
      sred[0][threadIdx.x >> 5] = vdisp;
      sred[1][threadIdx.x >> 5] = vdev;
    }
  }
  __syncthreads();
  if (threadIdx.x < 2) {
    float mx = 0.f;
    for (int w = 0; w < (S >> 5); ++w) mx = fmaxf(mx, sred[threadIdx.x][w]);
    a.blkmax[2 * blockIdx.x + threadIdx.x] = mx <= 3.0e38f ? sqrt((double)mx) * (1.0 + 1e-6) : 1e300;
  }
}

// ---- Cartesian method (Sec. III.C "method pimd") ---------------------------
// Bead velocities v; the springs of Eq. (1) enter the kicks as forces
// F_s^(k) = -m w_n^2 (2 x^k - x^(k-1) - x^(k+1)) (cyclic); A is the free drift
// x += tA v; O (App. D) acts on every bead with one friction.  Thread task
// t = (al * 3 + d) * P + k as in the normal-mode kernel.
__device__ __forceinline__ double spring_force(const double *row, int k, int P, double mmw2) {
  const double xm = row[k == 0 ? P - 1 : k - 1], xp = row[k == P - 1 ? 0 : k + 1];
  return -mmw2 * (2.0 * row[k] - xm - xp);
}

__global__ void __launch_bounds__(256) k_step_cart_f64(StepArgs a) {
  extern __shared__ double sm[];
  const int P = a.P;
  const int tileLen = a.A * 3 * P;
  double *sX = sm;               // positions at the start of the step
  double *sN = sX + tileLen;     // new positions
  double *sE = sN + tileLen;     // PILE_L deviates, stream O1, per element
  double *sE2 = sE + tileLen;    // OBABO: stream O2 of the previous step
  double *sC = sE2 + tileLen;    // [A][3] new centroids (water skin check)
  __shared__ double sred[2][8];
  const int tile0 = blockIdx.x * a.A;
  const int na = min(a.A, a.N - tile0);
  const int len = na * 3 * P;
  const size_t base = (size_t)tile0 * 3 * P;
  for (int t = threadIdx.x; t < len; t += blockDim.x) sX[t] = a.x[base + t];
  const uint64_t step = (uint64_t)(*a.step + a.step_off);
  if (a.thermo && a.noise_pre) {   // one Philox draw per (atom, bead) serves the three components
    const bool o2 = a.integrator == 1 && !a.first;
    for (int t = threadIdx.x; t < na * P; t += blockDim.x) {
      const int al = t / P, k = t - al * P;
      const int e = al * 3 * P + k;
      gauss3(a.seed, (uint32_t)(tile0 + al), (uint32_t)k, kStreamO1, step, sE[e], sE[e + P], sE[e + 2 * P]);
      if (o2)
        gauss3(a.seed, (uint32_t)(tile0 + al), (uint32_t)k, kStreamO2, step - 1, sE2[e], sE2[e + P],
               sE2[e + 2 * P]);
    }
  }
  __syncthreads();
  const double c1 = __ldg(a.mt.c1), c2 = __ldg(a.mt.c2);
  for (int task = threadIdx.x; task < len; task += blockDim.x) {
    const int k = task % P;
    const int r = task / P;
    const int i = tile0 + r / 3;
    auto noise = [&](uint32_t stream, uint64_t st, const double *pre) {
      return a.noise_pre ? pre[task] : gauss1(a.seed, (uint32_t)i, (uint32_t)k, stream, st, r % 3);
    };
    const double f = a.F[base + task] + spring_force(sX + r * P, k, P, __ldg(a.mass_mm + i) * a.wn2);
    const double im = __ldg(a.inv_mm + i) * a.ifmass;
    const double c2s = c2 * __ldg(a.sigv + i);
    double v = a.v[base + task];
    if (a.fix_u) v -= a.fix_u[3 * k + r % 3];   // the previous step's fixcom
    double x = sX[task];
    if (a.integrator == 0) {
      v = fma(a.kick * im, f, v);
      x = fma(a.half, v, x);
      if (a.thermo) v = fma(c1, v, c2s * noise(kStreamO1, step, sE));
      x = fma(a.half, v, x);
    } else {
      const double kb = a.half * im;
      if (!a.first) {
        v = fma(kb, f, v);
        if (a.thermo) v = fma(c1, v, c2s * noise(kStreamO2, step - 1, sE2));
      }
      if (a.thermo) v = fma(c1, v, c2s * noise(kStreamO1, step, sE));
      v = fma(kb, f, v);
      x = fma(2.0 * a.half, v, x);
    }
    a.v[base + task] = v;
    a.x[base + task] = x;
    if (a.xi && i % 3 == 0) {
      const int c = r % 3;
      const double Lc = a.dbox ? a.dbox[c] : a.box[c], iLc = a.dbox ? a.dbox[3 + c] : a.invbox[c];
      a.xi[((size_t)i + c) * P + k] = fix_wrap(x, a.pos, (float)x, (float)iLc, fix_pos(Lc, a.pos));   // row 3 (i / 3) + c
    }
    sN[task] = x;
  }
  if (!a.blkmax) return;
  // neighbour-list skin check of the oxygens: centroid = bead mean
  __syncthreads();
  for (int t = threadIdx.x; t < na * 3; t += blockDim.x) {
    const double *row = sN + t * P;
    double sum = 0.0;
    for (int j = 0; j < P; ++j) sum += row[j];
    sC[t] = sum / P;
  }
  __syncthreads();
  double vdisp = 0.0, vdev = 0.0;
  for (int t = threadIdx.x; t < na * P; t += blockDim.x) {
    const int al = t / P, k = t % P;
    const int i = tile0 + al;
    if (i % 3) continue;
    const double c0 = sC[al * 3], cc1 = sC[al * 3 + 1], cc2 = sC[al * 3 + 2];
    const double *xs = sN + al * 3 * P;
    const double e0 = xs[k] - c0, e1 = xs[P + k] - cc1, e2 = xs[2 * P + k] - cc2;
    vdev = fmax(vdev, e0 * e0 + e1 * e1 + e2 * e2);
    if (k == 0) {
      const int m = i / 3;
      const double g0 = c0 - a.cref[3 * m], g1 = cc1 - a.cref[3 * m + 1], g2 = cc2 - a.cref[3 * m + 2];
      vdisp = fmax(vdisp, g0 * g0 + g1 * g1 + g2 * g2);
      a.ccur[3 * m] = c0;
      a.ccur[3 * m + 1] = cc1;
      a.ccur[3 * m + 2] = cc2;
    }
  }
  vdisp = warp_max(vdisp);
  vdev = warp_max(vdev);
  if ((threadIdx.x & 31) == 0) {
    sred[0][threadIdx.x >> 5] = vdisp;
    sred[1][threadIdx.x >> 5] = vdev;
  }
  __syncthreads();
  if (threadIdx.x < 2) {
    double mx = 0.0;
    for (int w = 0; w < (int)((blockDim.x + 31) / 32); ++w) mx = fmax(mx, sred[threadIdx.x][w]);
    a.blkmax[2 * blockIdx.x + threadIdx.x] = (mx == mx) ? sqrt(mx) : 1e300;
  }
}

// Closing kick of a call, Cartesian: B(h/2) with the springs (and the final
// O(h/2) of OBABO).
__global__ void __launch_bounds__(256) k_close_cart_f64(StepArgs a) {
  const int P = a.P;
  const size_t total = (size_t)a.N * 3 * P;
  const uint64_t step = (uint64_t)(*a.step + a.step_off);
  const double c1 = __ldg(a.mt.c1), c2 = __ldg(a.mt.c2);
  for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (size_t)gridDim.x * blockDim.x) {
    const int k = (int)(t % P);
    const size_t r = t / P;
    const int d = (int)(r % 3);
    const int i = (int)(r / 3);
    const double f = a.F[t] + spring_force(a.x + r * P, k, P, __ldg(a.mass_mm + i) * a.wn2);
    double v = a.v[t];
    if (a.fix_u) v -= a.fix_u[3 * k + d];   // the last step's fixcom
    v = fma(a.half * (__ldg(a.inv_mm + i) * a.ifmass), f, v);
    if (a.integrator == 1 && a.thermo)
      v = fma(c1, v, c2 * __ldg(a.sigv + i) * gauss1(a.seed, (uint32_t)i, (uint32_t)k, kStreamO2, step, d));
    a.v[t] = v;
  }
}

__global__ void k_advance(int64_t *step, int n) {
  if (threadIdx.x == 0 && blockIdx.x == 0) *step += n;
}

// Initial velocities of mode (or bead) k ~ N(0, P kB T / (mu_k m mvv2e)),
// noise stream 2.
__global__ void k_thermal_v(double *v, const double *sigv, const double *imu, uint64_t seed, int N, int P) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= N * P) return;
  const int i = t / P, k = t % P;
  double e0, e1, e2;
  gauss3(seed, (uint32_t)i, (uint32_t)k, kStreamInit, 0ull, e0, e1, e2);
  const double s = imu ? sigv[i] * sqrt(imu[k]) : sigv[i];
  v[((size_t)i * 3 + 0) * P + k] = s * e0;
  v[((size_t)i * 3 + 1) * P + k] = s * e1;
  v[((size_t)i * 3 + 2) * P + k] = s * e2;
}

// Layout changes between the host order [P][N][3] and the device order [N][3][P].
__global__ void k_pna_to_nap(const double *src, double *dst, int N, int P) {
  const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  const size_t total = (size_t)N * 3 * P;
  if (t >= total) return;
  const int k = (int)(t % P);
  const size_t ia = t / P;
  const int a = (int)(ia % 3);
  const size_t i = ia / 3;
  dst[t] = src[((size_t)k * N + i) * 3 + a];
}

__global__ void k_nap_to_pna(const double *src, double *dst, int N, int P) {
  const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  const size_t total = (size_t)N * 3 * P;
  if (t >= total) return;
  const int a = (int)(t % 3);
  const size_t ki = t / 3;
  const size_t i = ki % N;
  const int k = (int)(ki / N);
  dst[t] = src[(i * 3 + a) * P + k];
}

// --- host launchers --------------------------------------------------------
// Atoms per block of the normal-mode step: the smallest tile that fills its
// warps best (A P close to a multiple of 32, at most 128 per component), as
// long as the grid still has two blocks for every SM of the GPU.
int step_tile_atoms(int N, int P) {
  const int need = std::min(N, 304);
  int best = 1;
  double eff = 0.0;
  for (int A = 1; A <= std::max(1, 128 / P); ++A) {
    if (A > 1 && (N + A - 1) / A < need) break;
    const double e = (double)A * P / ((A * P + 31) / 32 * 32);
    if (e > 1.02 * eff) {
      eff = e;
      best = A;
    }
  }
  return best;
}

int step_threads(int A, int P) { return 3 * ((A * P + 31) / 32 * 32); }

static size_t step_smem_bytes(int A, int P) {
  const size_t rows = 3 * (size_t)A, AP = (size_t)A * P;
  return rows * 2 * fix_pairs(P) * sizeof(int4) * 2 +   // limbs of x and F
         (2 * 3 * AP + rows) * sizeof(long long) +      // rows, centroids
         4 * AP * sizeof(double) + 3 * rows * sizeof(int) + 3 * AP * sizeof(float);
}

static size_t cart_smem_bytes(int A, int P) { return ((size_t)4 * A * 3 * P + 3 * A) * sizeof(double); }

cudaError_t launch_step(const StepArgs &a0, int threads, cudaStream_t s) {
  const int grid = (a0.N + a0.A - 1) / a0.A;
  StepArgs a = a0;
  if (a.method == 1) {
    static int nsm = 0;   // SM count of the device (one GPU per process)
    if (!nsm) {
      int dev = 0;
      cudaGetDevice(&dev);
      if (cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || nsm < 1) nsm = 152;
    }
    a.noise_pre = grid >= 4 * nsm ? 1 : 0;
    k_step_cart_f64<<<grid, threads, cart_smem_bytes(a.A, a.P), s>>>(a);
    return cudaGetLastError();
  }
  const size_t smem = step_smem_bytes(a.A, a.P);
  if (a.kspring && a.integrator == 0)
    k_step_f64<0, false, true><<<grid, threads, smem, s>>>(a);
  else if (a.kspring)
    k_step_f64<0, true, true><<<grid, threads, smem, s>>>(a);
  else if (a.integrator == 0)
    k_step_f64<0, false, false><<<grid, threads, smem, s>>>(a);
  else if (a.phase == 1)
    k_step_f64<1, true, false><<<grid, threads, smem, s>>>(a);
  else if (a.phase == 2)
    k_step_f64<2, true, false><<<grid, threads, smem, s>>>(a);
  else
    k_step_f64<0, true, false><<<grid, threads, smem, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_close(const StepArgs &a, int threads, cudaStream_t s) {
  if (a.method == 1) {
    const size_t total = (size_t)a.N * 3 * a.P;
    k_close_cart_f64<<<(unsigned)std::min<size_t>((total + 255) / 256, 4096), 256, 0, s>>>(a);
    return cudaGetLastError();
  }
  const int grid = (a.N + a.A - 1) / a.A;
  const size_t smem = step_smem_bytes(a.A, a.P);
  if (a.kspring && a.integrator == 0)
    k_step_f64<3, false, true><<<grid, threads, smem, s>>>(a);
  else if (a.kspring)
    k_step_f64<3, true, true><<<grid, threads, smem, s>>>(a);
  else if (a.integrator == 0)
    k_step_f64<3, false, false><<<grid, threads, smem, s>>>(a);
  else
    k_step_f64<3, true, false><<<grid, threads, smem, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_advance(int64_t *step, int n, cudaStream_t s) {
  k_advance<<<1, 32, 0, s>>>(step, n);
  return cudaGetLastError();
}

cudaError_t launch_thermal_v(double *v, const double *sigv, const double *imu, uint64_t seed, int N, int P,
                             cudaStream_t s) {
  const int total = N * P;
  k_thermal_v<<<(total + 255) / 256, 256, 0, s>>>(v, sigv, imu, seed, N, P);
  return cudaGetLastError();
}

cudaError_t launch_pna_to_nap(const double *src, double *dst, int N, int P, cudaStream_t s) {
  const size_t total = (size_t)N * 3 * P;
  k_pna_to_nap<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(src, dst, N, P);
  return cudaGetLastError();
}

cudaError_t launch_nap_to_pna(const double *src, double *dst, int N, int P, cudaStream_t s) {
  const size_t total = (size_t)N * 3 * P;
  k_nap_to_pna<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(src, dst, N, P);
  return cudaGetLastError();
}

}  // namespace pimd
