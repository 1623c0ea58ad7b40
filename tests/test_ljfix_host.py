"""The fixed-point Lennard-Jones pair (csrc/ljfix.cuh), compiled for the host,
against decimal arithmetic with 60 digits on the same separations: force scales
from sigma far below the cutoff to cutoffs next to the power of two above them,
and reciprocal seeds up to two units in the last place off."""
import os
import shutil
import subprocess
from decimal import Decimal, getcontext

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2602_13553_gb300", "csrc")

HARNESS = r"""
#include <cmath>
#include <cstdio>
#include <cstring>
#include <stdint.h>
static int g_ulp = 0;
static float seed_off(float v) {
  for (int i = 0; i < (g_ulp < 0 ? -g_ulp : g_ulp); ++i) v = std::nextafterf(v, g_ulp < 0 ? 0.0f : 1e30f);
  return v;
}
#define PIMD_RCP(x) seed_off(1.0f / (x))
#include "ljfix.cuh"
// a line: ulp, eps, sig, rc, d0, d1, d2 (separations in units of 2^-50 A) ->
// taken in fixed point, energy and virial shares, force on j (3), Xi_aa (3)
int main() {
  double eps, sig, rc;
  long long d0, d1, d2;
  const double box[3] = {1000.0, 1000.0, 1000.0};
  while (std::scanf("%d %lf %lf %lf %lld %lld %lld", &g_ulp, &eps, &sig, &rc, &d0, &d1, &d2) == 7) {
    const pimd::LjFix p = pimd::lj_fix_setup(eps, sig, rc, box);
    const int64_t d[3] = {d0, d1, d2};
    pimd::LjSums s;
    const bool in = p.on && pimd::lj_fix_pair<true>(p, d, s);
    std::printf("%d %.17g %.17g", (int)in, p.us * pimd::fix_energy(s), p.ws * pimd::fix_sum(s.T));
    for (int c = 0; c < 3; ++c) std::printf(" %.17g", p.fs * pimd::fix_sum(s.f[c]));
    for (int c = 0; c < 3; ++c) std::printf(" %.17g", 0.5 * p.w3 * pimd::fix_sum(s.w[c]));
    std::printf("\n");
  }
}
"""


def cuda_include():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    return os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")


@pytest.fixture(scope="module")
def pairs(tmp_path_factory):
    d = tmp_path_factory.mktemp("ljfix")
    src = d / "pair.cpp"
    src.write_text(HARNESS)
    exe = d / "pair"
    subprocess.run(["g++", "-std=c++17", "-O1", "-I" + CSRC, "-I" + cuda_include(), str(src), "-o", str(exe)],
                   check=True)

    def run(rows):
        text = "\n".join("%d %.17g %.17g %.17g %d %d %d" % tuple(r) for r in rows) + "\n"
        out = subprocess.run([str(exe)], input=text, capture_output=True, text=True, check=True).stdout
        return np.array([[float(w) for w in line.split()] for line in out.splitlines()])
    return run


def exact(eps, sig, rc, d):
    """U / 2, W / 2, force on j (3) and Xi_aa / 2 (3), or None beyond the cutoff."""
    getcontext().prec = 60
    D = [Decimal(int(c)) / Decimal(2) ** 50 for c in d]
    r2 = sum(c * c for c in D)
    if not r2 < Decimal(rc) ** 2:
        return None
    s6 = (Decimal(sig) ** 2 / r2) ** 3
    fr = 24 * Decimal(eps) * (2 * s6 * s6 - s6) / r2
    return [2 * Decimal(eps) * (s6 * s6 - s6), fr * r2 / 2] + [fr * c for c in D] + [fr * c * c / 2 for c in D]


EPS = 6.7e-3
SCALES = [(3.166, 6.0), (3.166, 7.5), (3.166, 7.9), (3.166, 9.0), (3.166, 12.0), (3.166, 15.8), (3.166, 20.0),
          (3.166, 3.3), (3.0, 3.9), (1.0, 3.9), (0.5, 3.9), (1.0, 7.9), (0.5, 7.9), (1.0, 6.0)]


def sample(sig, rc, lo, n, rng, ulps=(0,)):
    """Separations of random direction, lo to 1 of the cutoff."""
    r = rc * rng.uniform(lo, 1.0, n)
    e = rng.normal(size=(n, 3))
    e /= np.linalg.norm(e, axis=1)[:, None]
    d = np.rint(r[:, None] * e * 2.0 ** 50).astype(np.int64)
    return [(u, EPS, sig, rc, *row) for row in d.tolist() for u in ulps]


@pytest.mark.parametrize("sig,rc", SCALES)
def test_reciprocal_headroom(pairs, sig, rc):
    """T = y^3 (C y^3 - 1) (the virial is 12 eps c6 T) on the upper nine tenths of
    the cutoff's range, seeds up to two units off: y carries 2^-60 of itself, T is
    kept to 2^-58, its double to 2^-53 of itself: 1e-15 (1 + T) with six times
    the first."""
    rows = sample(sig, rc, 0.1, 150, np.random.default_rng(1), (-2, -1, 0, 1, 2))
    got = pairs(rows)
    assert got[:, 0].sum() > 0.3 * len(rows)
    b = 0
    while 2.0 ** b < 1.01 * rc:
        b += 1
    e, s2 = 0, sig * sig / 4.0 ** b
    while e < 7 and s2 * 2.0 ** (e + 1) <= 3.17:
        e += 1
    unit = 12.0 * EPS * (s2 * 2.0 ** e) ** 3
    for row, g in zip(rows, got):
        ref = exact(*row[1:4], row[4:])
        if ref is None or not g[0]:
            continue
        err = abs(Decimal(g[2]) - ref[1])
        assert err <= Decimal(1e-15 * (unit + abs(g[2]))), (row, float(err / Decimal(unit)))


@pytest.mark.parametrize("lo,hi", [(0.1, 1.0), (0.85, 1.0)])
@pytest.mark.parametrize("sig,rc", SCALES)
def test_relative_error(pairs, sig, rc, lo, hi):
    """Energy, virial, force and Xi_aa of a single pair, near or far, against its
    own size (the repulsive and the attractive part added): r^2 is cut by up to
    3 2^-64 of the scale, which seven powers of it make 24 2^-64 / x; beyond that
    the six FP64 roundings of the constants and the conversion, 6 2^-53, hold the
    pair's own truncations (2^-55)."""
    rows = [r for r in sample(sig, rc, lo, 200, np.random.default_rng(2))]
    got = pairs(rows)
    x0 = 1.0
    while x0 < 1.01 * rc:
        x0 *= 2.0
    n = 0
    for row, g in zip(rows, got):
        ref = exact(*row[1:4], row[4:])
        if ref is None or not g[0]:
            continue
        n += 1
        r2 = sum((float(c) * 2.0 ** -50) ** 2 for c in row[4:])
        s6 = (sig * sig / r2) ** 3
        size = 24.0 * EPS * (2.0 * s6 * s6 + s6)
        bar = 6.0 * 2.0 ** -53 + 24.0 * 2.0 ** -64 / (r2 / x0 ** 2)
        for q, (a, b) in enumerate(zip(g[1:], ref)):
            scale = 0.5 * size if q in (0, 1) or q > 4 else size / r2 ** 0.5
            assert abs(Decimal(a) - b) <= Decimal(bar * scale), (row, q, float(abs(Decimal(a) - b)) / scale)
    assert n > 30
