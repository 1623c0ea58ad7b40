// split.cu -- the split-precision form of the PIMD step and forces.
//
// State: the ring-polymer centroid of every atom in FP64 (position xc and
// centroid-mode velocity v~_0), the beads as FP32 deviations d^j = x^j - xc
// and the internal-mode velocities v~_k (k >= 1) in FP32, forces in FP32.
// Because rows k >= 1 of the normal-mode matrix (Eq. A1) are orthogonal to
// the constant row, q~_k = (M x)_k = (M d)_k for k >= 1: the internal modes
// are transformed from the small deviations alone, so FP32 rounding acts on
// ~0.1 A quantities instead of on absolute coordinates.  FP64 is kept for
// the centroid's position/momentum accumulation (A and O of mode 0 and its
// kick) and, in the estimators, for the compensated sums.
//
// HBM per bead-atom and step: step kernel reads F, d, v~ (36 B) and writes
// d, v~ (24 B), plus 96 B per atom for xc, v~_0; force kernel reads d (12 B)
// and writes F (12 B).
#include "common.cuh"
#include "nbr.cuh"

namespace pimd {

// FP32 deviate of the same Philox words as gauss1 (component d = 0, 1, 2):
// u = (w >> 8 + 1/2) 2^-24, Box-Muller in FP32.
__device__ __forceinline__ float gauss1f(uint64_t seed, uint32_t atom, uint32_t mode, uint32_t stream,
                                         uint64_t step, int d) {
  const uint4 w = philox4x32_10(
      make_uint4(atom, (mode & 0xffffu) | (stream << 16), (uint32_t)step, (uint32_t)(step >> 32)),
      make_uint2((uint32_t)seed, (uint32_t)(seed >> 32)));
  const uint32_t wa = d < 2 ? w.x : w.z;
  const uint32_t wb = d < 2 ? w.y : w.w;
  const float s = 5.9604644775390625e-8f;  // 2^-24
  const float r = sqrtf(-2.0f * __logf(((float)(wa >> 8) + 0.5f) * s));
  const float ang = 2.0f * (((float)(wb >> 8) + 0.5f) * s);
  float sn, cs;
  sincospif(ang, &sn, &cs);
  return r * (d == 1 ? sn : cs);
}

// The three deviates of gauss1f for d = 0, 1, 2 from one Philox draw (the
// same words and the same FP32 arithmetic, so the same values).
__device__ __forceinline__ void gauss3f(uint64_t seed, uint32_t atom, uint32_t mode, uint32_t stream,
                                        uint64_t step, float &e0, float &e1, float &e2) {
  const uint4 w = philox4x32_10(
      make_uint4(atom, (mode & 0xffffu) | (stream << 16), (uint32_t)step, (uint32_t)(step >> 32)),
      make_uint2((uint32_t)seed, (uint32_t)(seed >> 32)));
  const float s = 5.9604644775390625e-8f;  // 2^-24
  const float r0 = sqrtf(-2.0f * __logf(((float)(w.x >> 8) + 0.5f) * s));
  const float r1 = sqrtf(-2.0f * __logf(((float)(w.z >> 8) + 0.5f) * s));
  float sn, cs, sn2, cs2;
  sincospif(2.0f * (((float)(w.y >> 8) + 0.5f) * s), &sn, &cs);
  sincospif(2.0f * (((float)(w.w >> 8) + 0.5f) * s), &sn2, &cs2);
  e0 = r0 * cs;
  e1 = r0 * sn;
  e2 = r1 * cs2;
}

__device__ __forceinline__ float warp_maxf(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_down_sync(0xffffffffu, v, o));
  return v;
}

__device__ __forceinline__ void rotatef(float &q, float &v, float c, float s_over_w, float w_s) {
  const float qn = fmaf(c, q, s_over_w * v);
  const float vn = fmaf(-w_s, q, c * v);
  q = qn;
  v = vn;
}


__device__ __forceinline__ float wrapf(double x, double L, double invL) {
  return L > 0.0 ? (float)(x - L * floor(x * invL)) : (float)x;
}

// Tasks as in the FP64 step: t = (al * 3 + c) * P + k.  Phase 1 (every
// task, FP32): F~_k, q~_k (k >= 1) and the internal-mode update; the k = 0
// slot keeps F~_0 for phase 2.  Phase 2: centroid tasks (al, c) in FP64 --
// kick, drift, O with an FP32 deviate, drift -- packed one per lane; and
// the inverse transform of the internal modes into new deviations.
// PT > 0 fixes the bead count at compile time (the index arithmetic of every
// element -- divisions by P and by 3 -- then reduces to shifts and multiplies,
// which matter in this issue-bound kernel); PT = 0 reads it from the arguments.
template <int PT>
__global__ void __launch_bounds__(256) k_step_split(SplitStepArgs a) {
  extern __shared__ float smf[];
  const int P = PT > 0 ? PT : a.P;
  const int tileLen = a.A * 3 * P;
  float *sD = smf;
  float *sV = sD + tileLen;
  float *sF = sV + tileLen;
  float *sQ = sF + tileLen;
  float *sE = sQ + tileLen;      // PILE_L deviates of this step (stream O1), per element
  float *sE2 = sE + tileLen;     // OBABO: stream O2 of the previous step
  __shared__ float sred[2][8];
  const int tile0 = blockIdx.x * a.A;
  const int na = min(a.A, a.N - tile0);
  const int len = na * 3 * P;
  const size_t base = (size_t)tile0 * 3 * P;
  // d and F staged folded (u_j = x_j + x_{P-j}, u_{P-j} = x_j - x_{P-j}):
  // the forward transforms then sum one half of a row (rows of M are even
  // for modes k <= H = P/2, odd above), as in the FP64 step kernel
  const int H = P >> 1;
  // a harmonic well's F~_k is -k q~_k: neither read nor transformed
  const bool harm = a.kspring != nullptr;
  for (int t = threadIdx.x; t < len; t += blockDim.x) {
    const int j = t % P, pj = j == 0 ? 0 : P - j;
    const size_t g = base + t, gp = g - j + pj;
    const float da = a.d[g], fa = harm ? 0.f : a.F[g];
    float du = da, fu = fa;
    if (pj != j) {
      const float db = a.d[gp], fb = harm ? 0.f : a.F[gp];
      du = j < pj ? da + db : db - da;
      fu = j < pj ? fa + fb : fb - fa;
    }
    sD[t] = du;
    sV[t] = a.vk[g];
    sF[t] = fu;
  }
  const uint64_t step = (uint64_t)(*a.step + a.step_off);
  // one Philox draw per (atom, mode) serves the three components
  const bool o2 = a.integrator == 1 && !a.first;
  if (a.thermo) {
    for (int t = threadIdx.x; t < na * P; t += blockDim.x) {
      const int al = t / P, k = t - al * P;
      const int e = al * 3 * P + k;
      gauss3f(a.seed, (uint32_t)(tile0 + al), (uint32_t)k, kStreamO1, step, sE[e], sE[e + P], sE[e + 2 * P]);
      if (o2)
        gauss3f(a.seed, (uint32_t)(tile0 + al), (uint32_t)k, kStreamO2, step - 1, sE2[e], sE2[e + P],
                sE2[e + 2 * P]);
    }
  }
  __syncthreads();
  const float *__restrict__ Tf = a.Tff;
  const float kick = (float)a.kick, half = (float)a.half;
  for (int task = threadIdx.x; task < len; task += blockDim.x) {
    const int k = task % P;
    const int r = task / P;
    const int c = r % 3;
    const int i = tile0 + r / 3;
    const bool even = k <= H;
    const int n = even ? H + 1 : P - H - 1;
    const float *fx = sF + r * P + (even ? 0 : H + 1);
    const float *xx = sD + r * P + (even ? 0 : H + 1);
    const float *tf = Tf + k;
    float fa = 0.f, fb = 0.f, qa = 0.f, qb = 0.f;
    int j = 0;
    if (harm) {
      for (; j + 1 < n; j += 2) {
        qa = fmaf(__ldg(tf + j * P), xx[j], qa);
        qb = fmaf(__ldg(tf + (j + 1) * P), xx[j + 1], qb);
      }
      if (j < n) qa = fmaf(__ldg(tf + j * P), xx[j], qa);
    } else {
      for (; j + 1 < n; j += 2) {
        const float m0 = __ldg(tf + j * P), m1 = __ldg(tf + (j + 1) * P);
        fa = fmaf(m0, fx[j], fa);
        fb = fmaf(m1, fx[j + 1], fb);
        qa = fmaf(m0, xx[j], qa);
        qb = fmaf(m1, xx[j + 1], qb);
      }
      if (j < n) {
        const float m0 = __ldg(tf + j * P);
        fa = fmaf(m0, fx[j], fa);
        qa = fmaf(m0, xx[j], qa);
      }
    }
    float q = qa + qb;
    const float f = harm ? -(float)__ldg(a.kspring + i) * q : fa + fb;
    if (k == 0) {
      sQ[task] = f;      // F~_0, consumed by the centroid task below
      continue;
    }
    float v = sV[task];
    const float im = (float)__ldg(a.inv_mm + i);
    const float cA = __ldg(a.cAf + k), sA = __ldg(a.sAf + k), wsA = __ldg(a.wsAf + k);
    const float c1 = __ldg(a.c1f + k), c2s = __ldg(a.c2f + k) * (float)__ldg(a.sigv + i);
    if (a.integrator == 0) {
      v = fmaf(kick * im, f, v);
      rotatef(q, v, cA, sA, wsA);
      if (a.thermo) v = fmaf(c1, v, c2s * sE[task]);
      rotatef(q, v, cA, sA, wsA);
    } else {
      const float kb = half * im;
      if (!a.first) {
        v = fmaf(kb, f, v);
        if (a.thermo) v = fmaf(c1, v, c2s * sE2[task]);
      }
      if (a.thermo) v = fmaf(c1, v, c2s * sE[task]);
      v = fmaf(kb, f, v);
      rotatef(q, v, cA, sA, wsA);
    }
    sQ[task] = q;
    a.vk[base + task] = v;
  }
  __syncthreads();
  // centroid tasks, FP64: q~_0 = sqrt(P) xc, so drift is xc += tA v~_0 / sqrt(P)
  const double rsp = rsqrt((double)P);
  for (int t = threadIdx.x; t < na * 3; t += blockDim.x) {
    const int al = t / 3, c = t % 3;
    const int i = tile0 + al;
    const size_t ic = (size_t)i * 3 + c;
    double x = a.xc[ic], v = a.v0[ic];
    const double im = __ldg(a.inv_mm + i);
    const double f0 = harm ? -__ldg(a.kspring + i) * x / rsp : (double)sQ[t * P];   // q~_0 = sqrt(P) xc
    const double dr = a.tA * rsp;
    if (a.integrator == 0) {
      v = fma(a.kick * im, f0, v);
      x = fma(dr, v, x);
      if (a.thermo) v = fma(a.c1_0, v, a.c2_0 * __ldg(a.sigv + i) * (double)sE[t * P]);
      x = fma(dr, v, x);
    } else {
      const double kb = a.half * im;
      if (!a.first) {
        v = fma(kb, f0, v);
        if (a.thermo) v = fma(a.c1_0, v, a.c2_0 * __ldg(a.sigv + i) * (double)sE2[t * P]);
      }
      if (a.thermo) v = fma(a.c1_0, v, a.c2_0 * __ldg(a.sigv + i) * (double)sE[t * P]);
      v = fma(kb, f0, v);
      x = fma(dr, v, x);
    }
    a.xc[ic] = x;
    a.v0[ic] = v;
    if (a.xcw) a.xcw[ic] = wrapf(x, a.box[c], a.invbox[c]);
    sQ[t * P] = 0.f;   // the deviations carry no centroid mode
  }
  __syncthreads();
  // inverse, first half: C_j (bead j <= H, even modes) or S_{P-j} (bead
  // j > H, odd modes) into sF, free since the forward pass
  const float *__restrict__ Ti = a.Tif;
  for (int task = threadIdx.x; task < len; task += blockDim.x) {
    const int j = task % P;
    const bool even = j <= H;
    const int n = even ? H + 1 : P - H - 1;
    const float *qq = sQ + (task - j) + (even ? 0 : H + 1);
    const float *ti = Ti + j;
    float xa = 0.f, xb = 0.f;
    int k = 0;
    for (; k + 1 < n; k += 2) {
      xa = fmaf(__ldg(ti + k * P), qq[k], xa);
      xb = fmaf(__ldg(ti + (k + 1) * P), qq[k + 1], xb);
    }
    if (k < n) xa = fmaf(__ldg(ti + k * P), qq[k], xa);
    sF[task] = xa + xb;
  }
  __syncthreads();
  // second half: d'_j = C_j + S_j (j <= H), d'_{P-j} = C_j - S_j
  for (int task = threadIdx.x; task < len; task += blockDim.x) {
    const int j = task % P, pj = j == 0 ? 0 : P - j;
    const int row0 = task - j;
    const float dn = j <= H ? sF[task] + (pj > H ? sF[row0 + pj] : 0.f) : sF[row0 + pj] - sF[task];
    a.d[base + task] = dn;
    sD[task] = dn;
  }
  if (!a.blkmax) return;
  __syncthreads();
  // neighbour-list skin check of the oxygens: bead spread |d^k| and centroid
  // drift, squared and reduced in FP32 (the FP64 pipe is the scarce one; a
  // relative margin below keeps the bound conservative)
  float vdisp = 0.f, vdev = 0.f;
  for (int t = threadIdx.x; t < na * P; t += blockDim.x) {
    const int al = t / P, k = t % P;
    const int i = tile0 + al;
    if (i % 3) continue;
    const float *ds = sD + al * 3 * P;
    const float e0 = ds[k], e1 = ds[P + k], e2 = ds[2 * P + k];
    vdev = fmaxf(vdev, e0 * e0 + e1 * e1 + e2 * e2);
    if (k == 0) {
      const int m = i / 3;
      const double c0 = a.xc[3 * (size_t)i], c1 = a.xc[3 * (size_t)i + 1], c2 = a.xc[3 * (size_t)i + 2];
      const float g0 = (float)(c0 - a.cref[3 * m]), g1 = (float)(c1 - a.cref[3 * m + 1]);
      const float g2 = (float)(c2 - a.cref[3 * m + 2]);
      vdisp = fmaxf(vdisp, g0 * g0 + g1 * g1 + g2 * g2);
      a.ccur[3 * m] = c0;
      a.ccur[3 * m + 1] = c1;
      a.ccur[3 * m + 2] = c2;
    }
  }
  // NaN positions force a rebuild
  if (vdisp != vdisp) vdisp = __int_as_float(0x7f800000);
  if (vdev != vdev) vdev = __int_as_float(0x7f800000);
  vdisp = warp_maxf(vdisp);
  vdev = warp_maxf(vdev);
  if ((threadIdx.x & 31) == 0) {
    sred[0][threadIdx.x >> 5] = vdisp;
    sred[1][threadIdx.x >> 5] = vdev;
  }
  __syncthreads();
  if (threadIdx.x < 2) {
    float mx = 0.f;
    for (int w = 0; w < (int)((blockDim.x + 31) / 32); ++w) mx = fmaxf(mx, sred[threadIdx.x][w]);
    // margins for FP32 rounding of the deviations and of the squares
    a.blkmax[2 * blockIdx.x + threadIdx.x] = mx <= 3.0e38f ? sqrt((double)mx) * (1.0 + 1e-6) + 1e-4 : 1e300;
  }
}

// Closing B(h/2) (and O(h/2) for OBABO) of a call's last step.
__global__ void __launch_bounds__(256) k_close_split(SplitStepArgs a) {
  extern __shared__ float smf[];
  const int P = a.P;
  float *sF = smf;
  const int tile0 = blockIdx.x * a.A;
  const int na = min(a.A, a.N - tile0);
  const int len = na * 3 * P;
  const size_t base = (size_t)tile0 * 3 * P;
  for (int t = threadIdx.x; t < len; t += blockDim.x) sF[t] = a.F[base + t];
  __syncthreads();
  const uint64_t step = (uint64_t)(*a.step + a.step_off);
  const float *__restrict__ Mt = a.Mtf;
  for (int task = threadIdx.x; task < len; task += blockDim.x) {
    const int k = task % P;
    const int r = task / P;
    const int c = r % 3;
    const int i = tile0 + r / 3;
    const float *fx = sF + r * P;
    float fa = 0.f, fb = 0.f;
    int j = 0;
    for (; j + 1 < P; j += 2) {
      fa = fmaf(__ldg(Mt + j * P + k), fx[j], fa);
      fb = fmaf(__ldg(Mt + (j + 1) * P + k), fx[j + 1], fb);
    }
    if (j < P) fa = fmaf(__ldg(Mt + j * P + k), fx[j], fa);
    const float f = fa + fb;
    if (k == 0) {
      const size_t ic = (size_t)i * 3 + c;
      double v = fma(a.half * __ldg(a.inv_mm + i), (double)f, a.v0[ic]);
      if (a.integrator == 1 && a.thermo)
        v = fma(a.c1_0, v, a.c2_0 * __ldg(a.sigv + i) *
                               (double)gauss1f(a.seed, (uint32_t)i, 0u, kStreamO2, step, c));
      a.v0[ic] = v;
      continue;
    }
    float v = fmaf((float)a.half * (float)__ldg(a.inv_mm + i), f, a.vk[base + task]);
    if (a.integrator == 1 && a.thermo) {
      const float c1 = __ldg(a.c1f + k), c2s = __ldg(a.c2f + k) * (float)__ldg(a.sigv + i);
      v = fmaf(c1, v, c2s * gauss1f(a.seed, (uint32_t)i, (uint32_t)k, kStreamO2, step, c));
    }
    a.vk[base + task] = v;
  }
}

// --- forces -----------------------------------------------------------------

__global__ void __launch_bounds__(256) k_force_harmonic_split(SplitForceArgs a) {
  __shared__ double sU[256], sW[256];
  const int P = a.P;
  const int per = blockDim.x / P;
  const int i = blockIdx.x * per + threadIdx.x / P;
  const int k = threadIdx.x % P;
  float u = 0.f, w = 0.f;
  if (threadIdx.x < per * P && i < a.N) {
    const float ks = (float)__ldg(a.kspring + i);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const size_t id = ((size_t)i * 3 + c) * P + k;
      const float x = (float)a.xc[(size_t)i * 3 + c] + a.d[id];
      const float f = -ks * x;
      a.F[id] = f;
      u = fmaf(0.5f * ks * x, x, u);
      w = fmaf(x, f, w);
    }
  }
  sU[threadIdx.x] = u;
  sW[threadIdx.x] = w;
  __syncthreads();
  const int groups = min(per, a.N - blockIdx.x * per);
  for (int kk = threadIdx.x; kk < P; kk += blockDim.x) {
    double su = 0.0, sw = 0.0;
    for (int g = 0; g < groups; ++g) {
      su += sU[g * P + kk];
      sw += sW[g * P + kk];
    }
    a.Upart[(size_t)blockIdx.x * P + kk] = su;
    a.Wpart[(size_t)blockIdx.x * P + kk] = sw;
  }
  if (a.step_inc && blockIdx.x == 0 && threadIdx.x == 0) *a.step_inc += a.inc;
}

__device__ __forceinline__ float micf(float d, float L, float invL) { return fmaf(-rint_mul(d, invL), L, d); }

// FP32 sum with its rounding errors kept (Knuth's two-sum; intrinsics, so that no
// product is contracted into one of its additions): the FP64 pipe would take two
// slots a term.
struct FloatPair {
  float h, l;
  __device__ __forceinline__ void add(float x) {
    const float t = __fadd_rn(h, x), z = __fadd_rn(t, -h);
    l += __fadd_rn(__fadd_rn(h, -__fadd_rn(t, -z)), __fadd_rn(x, -z));
    h = t;
  }
  __device__ __forceinline__ void add(const FloatPair &o) {
    add(o.h);
    l += o.l;
  }
  // + a b, unrounded
  __device__ __forceinline__ void fma(float a, float b) {
    const float p = __fmul_rn(a, b);
    add(p);
    l += fmaf(a, b, -p);
  }
  __device__ __forceinline__ void half() {
    h *= 0.5f;
    l *= 0.5f;
  }
  __device__ __forceinline__ double value() const { return (double)h + (double)l; }
};

// Water-like model in FP32.  Work as in the FP64 kernel: a unit is one molecule
// and a chunk of Bk = min(P, 32) beads (G = 32 / Bk molecules where the beads
// leave lanes free), beads in adjacent lanes.  Many units: one warp each, four
// to a block; otherwise a block per unit, whose list `split` warps share and one
// more takes the bonds and the angle.  A pair vector is the minimum-image
// difference of the wrapped FP32 centroids plus the difference of the FP32
// deviations.  Candidates go two at a time on packed FP32 (each element rounds
// as a scalar would) and are summed one by one, in bucket and index order: the
// sums of a warp depend on the interacting pairs alone, not on the list's age.
//
// What bounds it is the latency of the gathers: the rows of the next two
// candidates are requested before the arithmetic of these.  No FP64 instruction
// is left but the list build's and four at the end: constants come converted,
// the list check compares in FP32, U and Tr Xi are sums of FP32 terms with their
// rounding errors kept (plain FP32 chains were 3e-8 of the sum off and 1% of a pass
// faster).  80 FP64 instructions a warp held 22 of 35.6 us at 512 molecules x 64
// beads and 5 of 13.4 at 216 x 20; now 15.0 and 7.8 us.
template <bool kSplit>
__global__ void __launch_bounds__(kSplit ? 256 : 128) k_force_water_split(SplitForceArgs a, int split) {
  extern __shared__ __align__(16) unsigned char fsm[];
  const int P = a.P;
  const int Bk = P < 32 ? P : 32, G = 32 / Bk;
  const int NS = kLJWarps * a.nb.groups;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int unit = kSplit ? blockIdx.x : blockIdx.x * 4 + warp;
  const int role = kSplit ? warp : 0;   // 0 .. split - 1: the list; then bonds and angle
  const int nmg = (a.nmol + G - 1) / G;
  const int chunk = unit / nmg, mg = unit - chunk * nmg;
  const int u = lane / Bk, kl = lane - u * Bk;
  const int m = mg * G + u, k = chunk * Bk + kl;
  const bool on = u < G && m < a.nmol && k < P;   // (a last block's spare warps have k >= P)
  int *s_nl = reinterpret_cast<int *>(fsm);             // [G][kMaxNeighbours]
  int *s_off = s_nl + G * kMaxNeighbours;               // [G][NS + 1]
  bool own = false;
  if (kSplit && a.check_nbr && role < split) {
    own = skin_exceeded(a.nb.blkmax, a.nb.nblk_check, a.nb.skin, 32 * split);
    if (own) {
      double Ld[3], iLd[3];
      list_box(a.nb, Ld, iLd);
      for (int q = warp; q < G; q += split) {
        const int mm = mg * G + q;
        if (mm >= a.nmol) break;
        int *nl = s_nl + q * kMaxNeighbours, *off = s_off + q * (NS + 1);
        const int total = list_molecule(a.nb, Ld, iLd, mm, NS, nl, off);
        if (chunk == 0) keep_list(a.nb, mm, NS, total, nl, off);
      }
      block_part_sync(32 * split);
    }
  }
  const float *const L = a.ff.L, *const iL = a.ff.iL;
  float F[9];
#pragma unroll
  for (int c = 0; c < 9; ++c) F[c] = 0.f;
  FloatPair U{0.f, 0.f}, W{0.f, 0.f};   // U and Tr Xi of the list (twice this molecule's)
  float bu = 0.f, bw = 0.f, au = 0.f, aw = 0.f;   // of the bonds, of the angle
  float co[3] = {0.f, 0.f, 0.f}, dO[3] = {0.f, 0.f, 0.f};
  if (on) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      co[c] = a.xcw[9 * m + c];
      dO[c] = a.d[(size_t)(9 * m + c) * P + k];
    }
  }
  if (on && role < split) {
    const int *off = own ? s_off + u * (NS + 1) : a.nb.off + (size_t)m * (NS + 1);
    const int *nl = own ? s_nl + u * kMaxNeighbours : a.nb.nbr + (size_t)m * kMaxNeighbours;
    int q = off[kSplit ? role * NS / split : 0];
    const int q1 = off[kSplit ? (role + 1) * NS / split : NS];
    const float rc2 = a.ff.rc2, e4 = a.ff.e4, e24 = a.ff.e24;
    const float2 sig2 = make_float2(a.ff.sig2, a.ff.sig2);
    const float2 e4v = make_float2(e4, e4), ne4 = make_float2(-e4, -e4);
    const float2 e48 = make_float2(2.f * e24, 2.f * e24), ne24 = make_float2(-e24, -e24);
    struct Cand { float c[2][3], d[2][3]; };
    auto load = [&](int j0, int j1, Cand &v) {
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        v.c[0][c] = __ldg(a.xcw + 9 * j0 + c);
        v.c[1][c] = __ldg(a.xcw + 9 * j1 + c);
        v.d[0][c] = __ldg(a.d + (size_t)(9 * j0 + c) * P + k);
        v.d[1][c] = __ldg(a.d + (size_t)(9 * j1 + c) * P + k);
      }
    };
    Cand cur, nxt;
    // a list's odd end pairs its last candidate with itself, masked
    if (q < q1) load(nl[q], nl[min(q + 1, q1 - 1)], cur);
#pragma unroll 1
    for (; q < q1; q += 2) {
      if (q + 2 < q1) load(nl[q + 2], nl[min(q + 3, q1 - 1)], nxt);
      float2 d[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        float2 e = make_float2(cur.c[0][c] - co[c], cur.c[1][c] - co[c]);
        e = __ffma2_rn(rint_mul2(e, make_float2(iL[c], iL[c])), make_float2(-L[c], -L[c]), e);
        d[c] = __fadd2_rn(e, make_float2(cur.d[0][c] - dO[c], cur.d[1][c] - dO[c]));
      }
      const float2 r2 = __ffma2_rn(d[2], d[2], __ffma2_rn(d[1], d[1], __fmul2_rn(d[0], d[0])));
      const bool i0 = r2.x < rc2, i1 = r2.y < rc2 && q + 1 < q1;
      if (i0 || i1) {
        // a candidate outside the cutoff gets 1 / r^2 = 0: it adds exact zeros
        const float2 inv = make_float2(i0 ? __frcp_rn(r2.x) : 0.f, i1 ? __frcp_rn(r2.y) : 0.f);
        const float2 s2 = __fmul2_rn(sig2, inv);
        const float2 s6 = __fmul2_rn(__fmul2_rn(s2, s2), s2);
        const float2 u = __ffma2_rn(e4v, s6, ne4);
        const float2 fr = __fmul2_rn(__fmul2_rn(__ffma2_rn(e48, s6, ne24), s6), inv);
        // one chain in list order: the zeros leave no trace of the list's other
        // candidates, or of which two were taken together
        U.fma(s6.x, u.x);
        U.fma(s6.y, u.y);
        W.fma(fr.x, i0 ? r2.x : 0.f);
        W.fma(fr.y, i1 ? r2.y : 0.f);
#pragma unroll
        for (int c = 0; c < 3; ++c) F[c] = fmaf(-fr.y, d[c].y, fmaf(-fr.x, d[c].x, F[c]));
      }
      cur = nxt;
    }
  }
  if (on && (!kSplit || role == split)) {
    float dv[2][3], r[2], ir[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const int row = 9 * m + 3 * (1 + h) + c;
        dv[h][c] = micf(a.xcw[row] - co[c], L[c], iL[c]) + (a.d[(size_t)row * P + k] - dO[c]);
      }
      r[h] = sqrtf(dv[h][0] * dv[h][0] + dv[h][1] * dv[h][1] + dv[h][2] * dv[h][2]);
      ir[h] = 1.f / r[h];
    }
    // bonds
    float fO[3] = {0.f, 0.f, 0.f};
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float dr = r[h] - a.ff.r0;
      bu = fmaf(0.5f * a.ff.kb * dr, dr, bu);
      const float g = -a.ff.kb * dr * ir[h];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const float fc = g * dv[h][c];
        F[3 + 3 * h + c] = fc;
        fO[c] -= fc;
        bw = fmaf(dv[h][c], fc, bw);
      }
    }
    // angle
    const float ir01 = ir[0] * ir[1];
    const float dot = dv[0][0] * dv[1][0] + dv[0][1] * dv[1][1] + dv[0][2] * dv[1][2];
    const float cth = fminf(1.f, fmaxf(-1.f, dot * ir01));
    const float th = acosf(cth);
    const float dth = th - a.ff.th0;
    const float pref = a.ff.kth * dth / sinf(th);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int g = 1 - h;
      const float ch = cth * ir[h] * ir[h];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const float fa = pref * fmaf(dv[g][c], ir01, -ch * dv[h][c]);
        F[3 + 3 * h + c] += fa;
        fO[c] -= fa;
        aw = fmaf(dv[h][c], fa, aw);
      }
    }
    au = 0.5f * a.ff.kth * dth * dth;
#pragma unroll
    for (int c = 0; c < 3; ++c) F[c] += fO[c];
  }
  if (a.step_inc && blockIdx.x == 0 && threadIdx.x == 0) *a.step_inc += a.inc;
  if (kSplit) {
    // partial sums of the warps, joined in order by the last warp
    float *sF = reinterpret_cast<float *>(s_off + ((G * (NS + 1) + 3) & ~3));   // [split][7][32]
    if (role < split) {
#pragma unroll
      for (int c = 0; c < 3; ++c) sF[(role * 7 + c) * 32 + lane] = F[c];
      sF[(role * 7 + 3) * 32 + lane] = U.h;
      sF[(role * 7 + 4) * 32 + lane] = U.l;
      sF[(role * 7 + 5) * 32 + lane] = W.h;
      sF[(role * 7 + 6) * 32 + lane] = W.l;
    }
    __syncthreads();
    if (role < split) return;
    float sum[3] = {0.f, 0.f, 0.f};
    for (int w = 0; w < split; ++w) {
#pragma unroll
      for (int c = 0; c < 3; ++c) sum[c] += sF[(w * 7 + c) * 32 + lane];
      U.add(FloatPair{sF[(w * 7 + 3) * 32 + lane], sF[(w * 7 + 4) * 32 + lane]});
      W.add(FloatPair{sF[(w * 7 + 5) * 32 + lane], sF[(w * 7 + 6) * 32 + lane]});
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) F[c] += sum[c];
  }
  U.half();
  W.half();
  U.add(bu);
  U.add(au);
  W.add(bw);
  W.add(aw);
  if (!on) return;
#pragma unroll
  for (int c = 0; c < 9; ++c) a.F[(size_t)(9 * m + c) * P + k] = F[c];
  a.Upart[(size_t)m * P + k] = U.value();
  a.Wpart[(size_t)m * P + k] = W.value();
}

// --- conversions between the split state and FP64 [N][3][P] arrays ----------

// x = xc + d, v~ (mode 0 from v~_0), F -> FP64
__global__ void k_expand_split(SplitStepArgs a, const float *F, double *x, double *v, double *Fd) {
  const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  const size_t total = (size_t)a.N * 3 * a.P;
  if (t >= total) return;
  const int k = (int)(t % a.P);
  const size_t ic = t / a.P;
  x[t] = a.xc[ic] + (double)a.d[t];
  v[t] = k == 0 ? a.v0[ic] : (double)a.vk[t];
  if (Fd) Fd[t] = (double)F[t];
}

// xc = bead average, d = x - xc, v~_0 and v~_k from FP64 [N][3][P] arrays; one
// lane group a row (at most four beads a lane).
__global__ void __launch_bounds__(128) k_compress_split(SplitStepArgs a, const double *x, const double *v) {
  const int P = a.P, W = row_lanes(P), l = threadIdx.x % W;
  const size_t ic = ((size_t)blockIdx.x * blockDim.x + threadIdx.x) / W;
  const bool on = ic < (size_t)a.N * 3;
  double xv[4], s = 0.0;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int k = l + q * W;
    xv[q] = on && k < P ? x[ic * P + k] : 0.0;
    s += xv[q];
  }
  const double xc = group_sum(s, W) / P;
  if (!on) return;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int k = l + q * W;
    if (k >= P) continue;
    a.d[ic * P + k] = (float)(xv[q] - xc);
    a.vk[ic * P + k] = k == 0 ? 0.f : (float)v[ic * P + k];
  }
  if (l) return;
  const int c = (int)(ic % 3);
  a.xc[ic] = xc;
  a.v0[ic] = v[ic * P];
  if (a.xcw) a.xcw[ic] = wrapf(xc, a.box[c], a.invbox[c]);
}

// --- host launchers ----------------------------------------------------------
size_t split_step_smem_bytes(int A, int P) { return (size_t)6 * A * 3 * P * sizeof(float); }

cudaError_t launch_step_split(const SplitStepArgs &a, int threads, cudaStream_t s) {
  const int grid = (a.N + a.A - 1) / a.A;
  const size_t smem = split_step_smem_bytes(a.A, a.P);
  switch (a.P) {
    case 8: k_step_split<8><<<grid, threads, smem, s>>>(a); break;
    case 16: k_step_split<16><<<grid, threads, smem, s>>>(a); break;
    case 32: k_step_split<32><<<grid, threads, smem, s>>>(a); break;
    case 64: k_step_split<64><<<grid, threads, smem, s>>>(a); break;
    case 128: k_step_split<128><<<grid, threads, smem, s>>>(a); break;
    default: k_step_split<0><<<grid, threads, smem, s>>>(a); break;
  }
  return cudaGetLastError();
}

cudaError_t launch_close_split(const SplitStepArgs &a, int threads, cudaStream_t s) {
  const int grid = (a.N + a.A - 1) / a.A;
  k_close_split<<<grid, threads, (size_t)a.A * 3 * a.P * sizeof(float), s>>>(a);
  return cudaGetLastError();
}

int force_blocks(int n_groups, int P);
int force_block_threads(int P);
int water_units(int nmol, int P);

// Warps that share a unit's neighbour list (ranges of buckets, as in FP64);
// 1: a warp takes whole units.  us a step, 1 against 2: 1024 units 32.1 against
// 30.4, 1400 units 33.1 against 37.2, 2048 units 38.4 against 43.2; 2 against 7:
// 600 units 27.6 against 28.4; 432 units 26.5 against 23.0; 4 against 7 at 432 units
// 23.6 against 23.0.
static int split_water_warps(int nmol, int P) {
  const int n = water_units(nmol, P);
  return n >= 1216 ? 1 : (n >= 512 ? 2 : 7);
}

// Whether the list check is a kernel of its own (the one-warp units).
bool split_lists_apart(int nmol, int P) { return split_water_warps(nmol, P) == 1; }

cudaError_t split_force_prepare() {   // a one-bead system's lists take more than 48 KB
  return cudaFuncSetAttribute(k_force_water_split<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024);
}

cudaError_t launch_force_split(const SplitForceArgs &a, bool water, cudaStream_t s) {
  if (water) {
    const int split = split_water_warps(a.nmol, a.P), units = water_units(a.nmol, a.P);
    if (split == 1) {
      k_force_water_split<false><<<(units + 3) / 4, 128, 0, s>>>(a, 1);
    } else {
      const int Bk = a.P < 32 ? a.P : 32, G = 32 / Bk, NS = kLJWarps * a.nb.groups;
      const size_t smem = (size_t)G * kMaxNeighbours * sizeof(int) +
                          (((size_t)G * (NS + 1) + 3) & ~(size_t)3) * sizeof(int) +
                          (size_t)split * 32 * 7 * sizeof(float);
      k_force_water_split<true><<<units, 32 * (split + 1), smem, s>>>(a, split);
    }
  } else
    k_force_harmonic_split<<<force_blocks(a.N, a.P), force_block_threads(a.P), 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_expand_split(const SplitStepArgs &a, const float *F, double *x, double *v, double *Fd,
                                cudaStream_t s) {
  const size_t total = (size_t)a.N * 3 * a.P;
  k_expand_split<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(a, F, x, v, Fd);
  return cudaGetLastError();
}

cudaError_t launch_compress_split(const SplitStepArgs &a, const double *x, const double *v,
                                  cudaStream_t s) {
  const size_t n = (size_t)a.N * 3 * row_lanes(a.P);
  k_compress_split<<<(unsigned)((n + 127) / 128), 128, 0, s>>>(a, x, v);
  return cudaGetLastError();
}

}  // namespace pimd
