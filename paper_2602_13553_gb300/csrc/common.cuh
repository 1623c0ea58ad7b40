// common.cuh -- device-side building blocks shared by the PIMD kernels:
// metal-unit constants, the Philox-4x32-10 generator, the Gaussian noise of
// the PILE_L O step, and the argument structs of every kernel.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "ljfix.cuh"
#include "noise64.cuh"

namespace pimd {

// Metal units (A, ps, eV, amu, K).  h and mvv2e are the values printed in
// App. C of the paper; Boltzmann's constant (not printed) is CODATA 2018.
constexpr double kBoltzmann = 8.617333262e-5;   // eV / K
constexpr double kPlanck = 4.135667403e-3;      // eV ps
constexpr double kMvv2e = 1.0364269e-4;         // eV per amu A^2 / ps^2
constexpr double kPi = 3.14159265358979323846;

constexpr int kMaxBeads = 128;
constexpr int kMaxNeighbours = 192;     // per molecule, O-O list with skin
// Neighbours are listed in NS = kLJWarps * groups buckets (j mod NS), which the
// force kernels deal to up to seven warps.
constexpr int kLJWarps = 14;

// Bits of the device error word (read back at synchronising calls).
enum : unsigned { kErrNbrOverflow = 1u, kErrNonFinite = 2u, kErrBoxSmall = 4u };

// Device barostat state (App. E), [kBaroWords] doubles, one v_W per box edge
// (the isotropic barostat keeps the three equal):
//   [0..2] v_W after the last completed sub-step
//   [3..5] v_W of this step's first A (after its B_W), [6..8] after its O
//   [9..11] box edges L, [12..14] 1 / L (the layout of ForceArgs::dbox)
//   [16..24], [25..33] factors of the centroid mode's A at those two v_W, for
//   each edge e^a, e^-a and (e^a - e^-a) / (2 v_W), a = tA v_W
enum {
  kBaroV = 0, kBaroVA1 = 3, kBaroVA2 = 6, kBaroL = 9, kBaroInvL = 12, kBaroA1 = 16, kBaroA2 = 25, kBaroWords = 36
};

// ---------------------------------------------------------------------------
// Philox-4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11): ten rounds of
//   (hi0, lo0) = M0 * c0, (hi1, lo1) = M1 * c2,
//   c <- (hi1 ^ c1 ^ k0, lo1, hi0 ^ c3 ^ k1, lo0),
// with the key bumped by the Weyl constants between rounds.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r) {
      k.x += 0x9E3779B9u;
      k.y += 0xBB67AE85u;
    }
    // 64-bit products: one multiply gives both halves
    const uint64_t p0 = (uint64_t)0xD2511F53u * c.x, p1 = (uint64_t)0xCD9E8D57u * c.z;
    c = make_uint4((uint32_t)(p1 >> 32) ^ c.y ^ k.x, (uint32_t)p1, (uint32_t)(p0 >> 32) ^ c.w ^ k.y, (uint32_t)p0);
  }
  return c;
}

// Noise streams of the counter's second word (bits 16..31).
enum : uint32_t { kStreamO1 = 0u, kStreamO2 = 1u, kStreamInit = 2u };

// The four words of (atom, normal mode, stream, step): counter = (atom,
// mode | stream << 16, step lo, step hi), key = seed.
__device__ __forceinline__ uint4 noise_words(uint64_t seed, uint32_t atom, uint32_t mode, uint32_t stream,
                                             uint64_t step) {
  return philox4x32_10(make_uint4(atom, (mode & 0xffffu) | (stream << 16), (uint32_t)step, (uint32_t)(step >> 32)),
                       make_uint2((uint32_t)seed, (uint32_t)(seed >> 32)));
}

// Three standard normal deviates of (atom, mode, stream, step): Box-Muller on
// u = (w + 1/2) 2^-32, (eta_x, eta_y) = r0 (cos, sin)(2 pi u1), eta_z = r1
// cos(2 pi u3), r = sqrt(-2 ln u).
__device__ __forceinline__ void gauss3(uint64_t seed, uint32_t atom, uint32_t mode, uint32_t stream,
                                       uint64_t step, double &e0, double &e1, double &e2) {
  const uint4 w = noise_words(seed, atom, mode, stream, step);
  const uint64_t r0 = bm_radius_fix(w.x), r1 = bm_radius_fix(w.z);
  int64_t sn, cs, s3, c3;
  bm_angle_fix(w.y, sn, cs);
  bm_angle_fix(w.w, s3, c3);
  e0 = bm_deviate(r0, cs);
  e1 = bm_deviate(r0, sn);
  e2 = bm_deviate(r1, c3);
}

// One standard normal deviate of the triple above (component d = 0, 1, 2),
// computed on its own so that one thread per component needs no exchange.
__device__ __forceinline__ double gauss1(uint64_t seed, uint32_t atom, uint32_t mode, uint32_t stream,
                                         uint64_t step, int d) {
  const uint4 w = noise_words(seed, atom, mode, stream, step);
  int64_t sn, cs;
  bm_angle_fix(d < 2 ? w.y : w.w, sn, cs);
  return bm_deviate(bm_radius_fix(d < 2 ? w.x : w.z), d == 1 ? sn : cs);
}

// Compensated running sum: (s, c) holds s + c, every addition keeping its
// rounding error in c (Neumaier's variant of Kahan summation), so a sum of
// many terms carries about one rounding of the total.  Plain aggregate
// (usable in shared memory); start from CSum{0.0, 0.0}.
struct CSum {
  double s, c;
  __device__ __forceinline__ void add(double x) {
    const double t = s + x;
    c += (fabs(s) >= fabs(x)) ? (s - t) + x : (x - t) + s;
    s = t;
  }
  __device__ __forceinline__ void add(const CSum &o) {
    add(o.s);
    c += o.c;
  }
  __device__ __forceinline__ double value() const { return s + c; }
};

// Warp-wide compensated sum (fixed shuffle tree); lane 0 holds the total.
__device__ __forceinline__ CSum warp_csum(CSum v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    CSum w{__shfl_down_sync(0xffffffffu, v.s, o), __shfl_down_sync(0xffffffffu, v.c, o)};
    v.add(w);
  }
  return v;
}

// Lanes per row: the smallest power of two >= min(P, 32).
__host__ __device__ __forceinline__ int row_lanes(int P) {
  int w = 1;
  while (w < P && w < 32) w <<= 1;
  return w;
}

__device__ __forceinline__ double group_sum(double v, int W) {
  for (int o = W >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// rint(x y), |x y| < 2^22, by the FP32 adder: rintf is an instruction of the
// special-function pipe (a warp in 8 clocks per SM partition).
constexpr float kRintMagic = 12582912.0f;   // 1.5 2^23
__device__ __forceinline__ float rint_mul(float x, float y) { return __fadd_rn(__fmaf_rn(x, y, kRintMagic), -kRintMagic); }
__device__ __forceinline__ float2 rint_mul2(float2 x, float2 y) {
  return __fadd2_rn(__ffma2_rn(x, y, make_float2(kRintMagic, kRintMagic)), make_float2(-kRintMagic, -kRintMagic));
}

// Minimum-image component (box edge L > 0; round half to even like rint).
__device__ __forceinline__ double mic(double d, double L, double invL) {
  return d - L * rint(d * invL);
}

// ---------------------------------------------------------------------------
// Kernel arguments.  Device layout of x, v, F: [N][3][P] (atom, component,
// bead/mode), i.e. every atom's P beads are contiguous per component.
// ---------------------------------------------------------------------------
struct ModeTables {
  const double *cA;    // [P] cos(w_k tA)
  const double *sA;    // [P] sin(w_k tA)/w_k   (tA for k = 0)
  const double *wsA;   // [P] w_k sin(w_k tA)   (0 for k = 0)
  const double *c1;    // [P] exp(-tO / tau_k)
  const double *c2;    // [P] sqrt(1 - c1^2) / sqrt(mu_k)  (noise of mode k)
  const double *lam;   // [P] lambda_k (Eq. A2)
  const double *mu;    // [P] fictitious-mass factor mu_k: m^(k) = mu_k m (fmmode, fmass)
  const double *imu;   // [P] 1 / mu_k
  // the folded transforms (H = floor(P/2)) in fixed point (fixed.cuh):
  // [fix_pairs(P)][P], limbs (h, l) of terms i = 2p and 2p + 1, scaled by
  // 2^(55 - fem).  Term i of mode k is M[k][i] (k <= H) or M[k][P - (H + 1 + i)]
  // (k > H; 0 past the row); of bead j, M[i][j] (j <= H) or M[H + 1 + i][P - j]
  const int4 *fTf, *fTi;
  int fem;
  // A(h/2) O(h) A(h/2) of BAOAB per mode, [6][P]: q' = m0 q + m1 v + m2 n,
  // v' = m3 q + m4 v + m5 n with n = sqrt(P kB T / (m mvv2e)) eta
  const double *map6;
  double rsp;          // 1 / sqrt(P)
};

struct StepArgs {
  int N, P, A;                 // atoms, beads, atoms per tile
  ModeTables mt;
  const double *inv_mm;        // [N] 1 / (m mvv2e)
  const double *kmm;           // [N] duration of this step's kick / (m mvv2e)
  int mu_one;                  // every imu_k is 1
  const double *sigv;          // [N] sqrt(P kB T / (m mvv2e))
  double *x;                   // [N][3][P] Cartesian positions
  double *v;                   // [N][3][P] normal-mode velocities
  const double *F;             // [N][3][P] Cartesian forces
  const double *kspring;       // normal modes in a harmonic well: [N] m mvv2e omega^2, F is not read; or null
  const int64_t *step;         // device step counter (step index of this step = *step + step_off)
  int step_off;
  long long *xi;               // water: [nmol][3][P] wrapped fixed-point positions of the oxygens, or null
  int pos;                     // their fraction bits (LjFix)
  double box[3], invbox[3];    // water
  const double *dbox;          // device box (barostat state at kBaroL), overriding box/invbox, or null
  // water-like systems: neighbour-list skin check of the oxygens (atoms 3m)
  const double *cref;          // [nmol][3] centroids at the last list build, or null
  double *ccur;                // [nmol][3] current centroids (written)
  double *blkmax;              // [gridDim.x][2] per-block max |c - cref| and max_k |x^k - c|
  double kick;                 // B before A: h/2 (first step of a call) or h (two merged halves)
  double half;                 // h/2
  int integrator;              // 0 BAOAB, 1 OBABO
  int first;                   // OBABO: 1 if no B+O of a previous step is pending
  int thermo;                  // 1 PILE_L
  uint64_t seed;
  // Cartesian method (v holds bead velocities): springs -m w_n^2 (2 x_k -
  // x_{k-1} - x_{k+1}) join the forces, bead masses fmass m; mt.c1/c2 hold
  // the one bead friction (tau = scale / (2 w_n)) and its noise factor
  int method;                  // 0 nmpimd, 1 pimd (Cartesian)
  double ifmass;               // 1 / fmass
  double wn2;                  // omega_n^2
  const double *mass_mm;       // [N] m mvv2e
  const double *baro;          // barostat state (centroid propagation under v_W), or null
  // OBABO with the barostat runs a step in two launches around the B_W that
  // needs the velocities after the O(h/2) sub-steps: phase 1 = the previous
  // step's closing B O and this step's O (velocities only), phase 2 = B(h/2)
  // A(h) and the new positions; phase 0 = the whole step in one launch
  int phase;
  const double *fix_u;         // fixcom of the previous step, still to be subtracted from v: [k][3], or null
  int noise_pre;               // Cartesian: 1: PILE_L deviates drawn once per (atom, bead) into shared memory
};

// B_W of the barostat (App. E) over a kick of length tB that starts from the
// current velocities, and, when a step follows, that step's v_W at its two A
// sub-steps (O_W in between) and the box they leave.
struct BaroArgs {
  int N, P, nmol;
  const double *x, *v, *F;     // [N][3][P]
  double rsp;                  // 1 / sqrt(P)
  const double *mass_mm, *inv_mm;   // [N] m^(0) mvv2e (fictitious masses included), and its inverse
  double invP;
  const double *Wpart;         // [nmol][P] Tr Xi rows of the force kernel
  const double *W3part;        // [nmol][P][3] diagonal Xi_aa rows (anisotropic), or null
  int axes;                    // 0: isotropic; else the mask of edges with their own v_W
  double *baro;
  double t0, tA;               // the B_W covers [t0, t0 + tB] of the kick that the next kernel applies
  int step_follows;
  // OBABO: the start-of-step call first applies the opening O_W (mode 0) and
  // scales the box once by exp(tA v_W), tA = h; the end-of-step call applies
  // the closing O_W (mode 1, keyed on the step just completed) after its B_W
  int obabo;
  double nkT, npext;           // n kB T; n P_ext
  // weights of B_W's three terms: 3 tB / W (per edge tB / W), tB^2 / W and
  // tB^3 / 3W, W = 3 n N kB T taup^2 (n N kB T taup^2 per edge)
  double k1, k2, k3;
  int thermo;
  double c1W, sigW;            // exp(-h / tau_0); c2 sqrt(n kB T / W)
  uint64_t seed;
  const int64_t *step;
  double Lmin;                 // smallest allowed box edge (2 rc)
  unsigned *err;
  const double *fix_u;         // fixcom still to be subtracted from v (centroid mode), or null
  double *part;                // partial sums (sums_part_doubles)
  unsigned *count;             // finished blocks, zero between launches
};

// fixcom: the centre-of-mass velocity of the centroid mode (normal modes) or
// of every bead (Cartesian) as it will stand after the closing B(h/2) that the
// next kernel applies (the removal belongs at the end of the step; subtracting
// its predicted value first is the same linear operation).
struct FixcomArgs {
  int N, P, method;
  const double *mass_mm;       // [N] m mvv2e
  double imsum;                // 1 / their sum
  double rsp;                  // 1 / sqrt(P)
  const double *x, *F, *v;     // [N][3][P]
  double *u;                   // out: [nb][3], subtracted by the next kernel
  double *part;                // partial sums (sums_part_doubles)
  unsigned *count;             // finished blocks, zero between launches
  double half;                 // h/2
  double imu0;                 // 1 / mu_0 (normal modes) or 1 / fmass (Cartesian)
  double wn2;                  // omega_n^2 (Cartesian springs)
  // OBABO with PILE_L: the closing O(h/2) follows the kick, v <- c1 v + c2 sigv eta
  int obabo_thermo;
  uint64_t seed;
  const int64_t *step;         // device counter, already advanced past this step
  const double *c1, *c2;       // [P] O tables (c2 includes 1 / sqrt(mu_k))
  const double *sigv;          // [N] sqrt(P kB T / (m mvv2e))
};

// O-O neighbour lists of a single water-like system (nbr.cuh).
struct NbrList {
  int nmol;
  const double *dbox;          // device box (barostat state at kBaroL), overriding box/invbox, or null
  double box[3], invbox[3];
  const double *ccur;          // [nmol][3] current centroids of the oxygens
  double *cref;                // [nmol][3] centroids at the last build (written on rebuild)
  const double *blkmax;        // [nblk_check][2] per-block max |c - cref|, max_k |x^k - c|
  int nblk_check;
  double skin, rlist;          // rlist = rc + skin
  int *nbr;                    // [nmol][kMaxNeighbours] neighbours grouped by bucket j mod NS
  int *off;                    // [nmol][NS + 1] bucket offsets into the molecule's row
  int groups;                  // NS = kLJWarps * groups buckets
  unsigned *err;
};

struct ForceArgs {
  int N, P, nmol;
  const double *x;             // [N][3][P]
  const int64_t *xi;           // water: [nmol][3][P] wrapped fixed-point positions of the oxygens
  LjFix lj;                    // water: fixed-point pairs
  int64_t *step_inc;           // if not null, block 0 advances the step counter by inc
  int inc;
  double *F;                   // [N][3][P]
  double *Upart, *Wpart;       // [rows][P] bead sums of U and Tr Xi (rows: blocks or molecules)
  double *W3part;              // water: [nmol][P][3] diagonal Xi_aa as well, or null
  const double *kspring;       // harmonic: [N] m mvv2e omega^2
  double kb, r0, kth, th0, eps, sig, rc;
  NbrList nb;
  // a small system's force blocks take the step's rebuild decision themselves
  // and list their molecules' neighbours before the pair loop
  int check_nbr;
};

// Split precision (split.cu): FP64 centroid xc, v~_0 [N][3]; FP32 deviations
// d = x - xc and internal-mode velocities v~_k (k >= 1) [N][3][P]; FP32 forces.
struct SplitStepArgs {
  int N, P, A;
  const float *Mtf;            // [P][P] FP32 copy of M^T
  const float *Tff, *Tif;      // [P/2 + 1][P] FP32 folded forward / inverse tables (terms as of ModeTables::fTf, fTi)
  const float *cAf, *sAf, *wsAf, *c1f, *c2f;   // FP32 mode coefficients (k >= 1)
  double tA, c1_0, c2_0;       // centroid: drift time of one A, O coefficients
  const double *inv_mm, *sigv; // [N]
  double *xc, *v0;             // [N][3]
  float *d, *vk;               // [N][3][P]
  const float *F;              // [N][3][P]
  const double *kspring;       // harmonic well: [N] m mvv2e omega^2, F is not read; or null
  float *xcw;                  // [N][3] centroids wrapped into the box, FP32 (water), or null
  double box[3], invbox[3];
  const int64_t *step;
  int step_off;
  const double *cref;          // water: [nmol][3] centroids at the last list build, or null
  double *ccur;
  double *blkmax;
  double kick, half;
  int integrator, first, thermo;
  uint64_t seed;
};

// The water-like model's constants in FP32 (rounded once on the host: an FP64
// conversion in the kernel costs a slot of the FP64 pipe in every warp).
struct SplitFF {
  float L[3], iL[3];
  float rc2, sig2, e4, e24;    // rc^2, sigma^2, 4 eps, 24 eps
  float kb, r0, kth, th0;
};

struct SplitForceArgs {
  int N, P, nmol;
  const double *xc;            // [N][3]
  const float *xcw;            // [N][3] wrapped FP32 centroids (water)
  const float *d;              // [N][3][P]
  float *F;                    // [N][3][P]
  double *Upart, *Wpart;
  int64_t *step_inc;           // if not null, block 0 advances the step counter by inc
  int inc;
  const double *kspring;
  SplitFF ff;                  // water
  NbrList nb;
  int check_nbr;               // as ForceArgs::check_nbr
};

// Columns of an estimator row: K, S, U and Tr Xi per mode or bead, then
// sum r.F, sum (r - r_c).F and m^(0) |v~_0|^2.
__host__ __device__ constexpr int est_columns(int P) { return 4 * P + 3; }

struct EstArgs {
  int N, P, A;
  int method;                  // 0 nmpimd, 1 pimd (Cartesian: v holds bead velocities)
  ModeTables mt;
  const double *mass_mm;       // [N] m mvv2e
  const double *x, *v, *F;
  double wn2;                  // omega_n^2
  int nblk_force;
  const double *Upart, *Wpart; // [nblk_force][P]
  double *part;                // [rows][est_columns(P)]
};

struct EstFinalArgs {
  int N, P, nblk_est;
  const double *part;          // [nblk_est][est_columns(P)]
  double *tot;                 // [est_columns(P)] column sums
  unsigned *count;             // finished blocks, zero between calls
  double kT, volume, kB;
  const double *dbox;          // device box edges (barostat): volume = L0 L1 L2, or null
  double *out;                 // [3P + 12]
  unsigned *err;
};

}  // namespace pimd
