"""The estimator reduction of the single-system handle against the oracle's
estimators of the same state, at the edges of its tiles and rows: one task,
partial tiles, more tiles than rows of partials, odd and maximal bead counts,
Cartesian beads, split precision."""
import math

import numpy as np
import pytest

from paper_2602_13553_gb300 import inputs
from tests._gpu import coord_err, pimd, scalar_err  # noqa: F401

pytestmark = pytest.mark.gpu

OMEGA_HO = 0.1 / (4.135667403e-3 / (2 * math.pi))

# Every output is a sum of products of the state, compensated on both sides
# or short: its rounding is that of q~ = M x (a sum of P terms, each within
# 2^-53 of |x| sqrt(2)) relative to the mode's own size, which at these inputs
# (thermal bead spread over ~1/10 of |x|) is below 128 * 10 * 2^-53 ~ 2e-13
# squared in S: 1e-11 leaves a factor of 20.
TOL = 1e-11


@pytest.mark.parametrize("N,P,method", [(1, 1, 0), (1, 128, 0), (7, 5, 0), (700, 1, 0), (613, 17, 0),
                                        (1300, 128, 0), (5, 2, 1), (40, 33, 1), (900, 96, 1)])
def test_estimators_match_oracle(orc, pimd, N, P, method):
    x0, mass = inputs.harmonic(N, P, seed=N + P, std=0.1)
    kw = dict(T=300.0, dt=2.5e-4, potential=0, ff=(OMEGA_HO,), seed=3, method=method)
    s = pimd.Simulation(x0, mass, **kw)
    s.step(3)
    x, v, _ = s.get_state()
    first, got = s.estimators(), s.estimators()
    s.close()
    want = orc.Sim(x, mass, v0=v, **kw).estimators()
    for k in ("K_mode", "S_mode", "U_bead"):
        assert coord_err(got[k], want[k]) < TOL, k
        assert np.array_equal(first[k], got[k]), k      # the second call sums alike
    for k in ("H", "K_VR", "K_CV", "T_ring"):
        assert scalar_err(got[k], want[k]) < TOL, k
    # K_PR is a difference of its kinetic term 3 P N kB T / 2 and the springs
    assert abs(got["K_PR"] - want["K_PR"]) < TOL * 1.5 * P * N * 8.617333262e-5 * 300.0


@pytest.mark.parametrize("N,P,method", [(1, 3, 0), (701, 8, 0), (333, 9, 1)])
def test_sums_over_a_wide_range(orc, pimd, N, P, method):
    """Kinetic terms over 24 decades, largest first, last and in between: every
    sum is rounded once, its terms within 2^-51 of themselves, so 1e-14 leaves
    a factor of 20."""
    x0, mass = inputs.harmonic(N, P, seed=N, std=0.1)
    g = np.random.default_rng(N + P)
    mass = mass * 10.0 ** g.uniform(-6.0, 6.0, N)
    v0 = g.standard_normal(x0.shape) * 10.0 ** g.uniform(-6.0, 6.0, (1, N, 1))
    kw = dict(T=300.0, dt=2.5e-4, potential=0, ff=(OMEGA_HO,), seed=3, method=method)
    s = pimd.Simulation(x0, mass, v0=v0, **kw)
    got = s.estimators()
    s.close()
    want = orc.Sim(x0, mass, v0=v0, **kw).estimators()
    assert coord_err(got["K_mode"], want["K_mode"]) < 1e-14
