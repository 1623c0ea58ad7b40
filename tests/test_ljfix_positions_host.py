"""Fixed-point positions of the Lennard-Jones pairs (csrc/ljfix.cuh), compiled for
the host: from FP64 coordinates through wrapping and minimum image to the pair's
force, against 60-digit decimals, side by side with the FP64 expressions."""
import subprocess
from decimal import Decimal, getcontext
from fractions import Fraction

import numpy as np
import pytest

from tests.test_ljfix_host import CSRC, EPS, cuda_include

HARNESS = r"""
#include <cmath>
#include <cstdio>
#include <stdint.h>
#include "ljfix.cuh"
// a line: sig, rc, L, x_i (3), x_j (3) -> taken in fixed point, force on j (3)
int main() {
  double sig, rc, L, x[2][3];
  while (std::scanf("%lf %lf %lf %lf %lf %lf %lf %lf %lf", &sig, &rc, &L, &x[0][0], &x[0][1], &x[0][2], &x[1][0],
                    &x[1][1], &x[1][2]) == 9) {
    const double box[3] = {L, L, L};
    const pimd::LjFix p = pimd::lj_fix_setup(EPS, sig, rc, box);
    const int64_t LQ = pimd::fix_pos(L, p.pos);
    int64_t d[3];
    for (int c = 0; c < 3; ++c) {
      int64_t w[2];
      for (int q = 0; q < 2; ++q) w[q] = pimd::fix_wrap(x[q][c], p.pos, (float)x[q][c], (float)(1.0 / L), LQ);
      d[c] = pimd::fix_mic(w[1] - w[0], LQ);
    }
    pimd::LjSums s;
    const bool in = p.on && pimd::lj_fix_pair<false>(p, d, s);
    std::printf("%d", (int)in);
    for (int c = 0; c < 3; ++c) std::printf(" %.17g", p.fs * pimd::fix_sum(s.f[c]));
    std::printf("\n");
  }
}
"""


@pytest.fixture(scope="module")
def forces(tmp_path_factory):
    d = tmp_path_factory.mktemp("ljpos")
    (d / "pos.cpp").write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-O1", "-DEPS=%r" % EPS, "-I" + CSRC, "-I" + cuda_include(),
                    str(d / "pos.cpp"), "-o", str(d / "pos")], check=True)

    def run(rows):
        text = "\n".join(" ".join("%.17g" % v for v in r) for r in rows) + "\n"
        out = subprocess.run([str(d / "pos")], input=text, capture_output=True, text=True, check=True).stdout
        return np.array([[float(w) for w in line.split()] for line in out.splitlines()])
    return run


@pytest.mark.parametrize("L,spread", [(12.42, 0), (24.84, 0), (13.0, 5), (200.0, 0), (255.5, 2), (300.0, 0),
                                      (2000.0, 0)])
def test_force_from_positions(forces, L, spread):
    """Oxygens uniform in a box around the origin, up to `spread` boxes away, pairs
    2.5 to 5.9 A apart: the rms error of the force (of its repulsive and attractive
    parts added) is no larger than that of the FP64 expressions."""
    getcontext().prec = 60
    rng = np.random.default_rng(int(L) + spread)
    sig, rc, n = 3.166, 6.0, 1500
    a = rng.uniform(-0.5, 0.5, (n, 3)) * L
    e = rng.normal(size=(n, 3))
    b = a + e / np.linalg.norm(e, axis=1)[:, None] * rng.uniform(2.5, 5.9, (n, 1))
    b -= L * np.rint(b / L)
    a += L * rng.integers(-spread, spread + 1, (n, 3))
    b += L * rng.integers(-spread, spread + 1, (n, 3))
    got = forces([(sig, rc, L, *p, *q) for p, q in zip(a, b)])
    assert got[:, 0].all()
    fix, f64 = [], []
    for p, q, g in zip(a, b, got):
        D = []
        for u, v in zip(p, q):
            f = Fraction(float(v)) - Fraction(float(u))
            f -= Fraction(L) * round(f / Fraction(L))
            D.append(Decimal(f.numerator) / Decimal(f.denominator))
        r2 = sum(c * c for c in D)
        s6 = (Decimal(sig) ** 2 / r2) ** 3
        fr = 24 * Decimal(EPS) * (2 * s6 * s6 - s6) / r2
        size = float(24 * Decimal(EPS) * (2 * s6 * s6 + s6) / r2.sqrt())
        d = q - p
        d = d - L * np.rint(d * (1.0 / L))
        R2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2]
        inv = 1.0 / R2
        s2 = sig * sig * inv
        S = s2 * s2 * s2
        f8 = 24.0 * EPS * (2.0 * S * S - S) * inv
        fix.append(float(sum((Decimal(x) - fr * c) ** 2 for x, c in zip(g[1:], D))) ** 0.5 / size)
        f64.append(float(sum((Decimal(f8 * x) - fr * c) ** 2 for x, c in zip(d, D))) ** 0.5 / size)
    rf, r8 = (np.sqrt(np.mean(np.square(v))) for v in (fix, f64))
    print("L = %g: fixed point %.2e, FP64 %.2e" % (L, rf, r8))
    assert rf <= r8
