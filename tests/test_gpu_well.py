"""Oscillators, whose steps form their own forces (F~ = -k q~) and whose step
counter advances once a call: against the oracle over call lengths on both sides
of a graph replay, and one long call against many short ones in FP64 and split
precision (whose bead counts are compared with the oracle in test_gpu_split)."""
import math

import numpy as np
import pytest

from paper_2602_13553_gb300 import inputs
from tests._gpu import coord_err, pimd  # noqa: F401
from tests.test_gpu_parity import _compare_est, _pair

pytestmark = pytest.mark.gpu

OMEGA_HO = 0.1 / (4.135667403e-3 / (2 * math.pi))


@pytest.mark.parametrize("integrator,thermostat,N,P,calls", [
    (0, 1, 30, 8, (1, 32, 33, 34, 70)), (1, 1, 30, 8, (1, 32, 33, 34, 70)), (0, 0, 7, 1, (2, 40)),
    (1, 0, 5, 33, (3,)), (0, 1, 400, 17, (5, 66)), (1, 1, 3, 128, (4,))])
def test_fp64(orc, pimd, integrator, thermostat, N, P, calls):
    x0, mass = inputs.harmonic(N, P, seed=N, std=0.1)
    mass = mass * (1.0 + np.arange(N) % 3)
    c, g = _pair(orc, pimd, x0, mass, T=300.0, dt=2.5e-4, potential=0, ff=(OMEGA_HO,), integrator=integrator,
                 thermostat=thermostat)
    for n in calls:
        c.run(n)
        g.step(n)
        x, v, st = g.get_state()
        assert st == sum(calls[:calls.index(n) + 1])
        assert coord_err(x, c.x) < 1e-10 and coord_err(v, c.v) < 1e-10
        _compare_est(g.estimators(), c.estimators(), 1e-10)


@pytest.mark.parametrize("precision", [0, 1])
def test_call_lengths_agree(pimd, precision):
    x0, mass = inputs.harmonic(50, 32, seed=2, std=0.1)
    kw = dict(T=300.0, dt=2.5e-4, potential=0, ff=(OMEGA_HO,), seed=4, precision=precision)
    a, b = pimd.Simulation(x0, mass, **kw), pimd.Simulation(x0, mass, **kw)
    a.step(100)
    for n in (1, 33, 32, 34):
        b.step(n)
    (xa, va, sa), (xb, vb, sb) = a.get_state(), b.get_state()
    assert sa == sb == 100
    # a call's end splits a kick into two halves: rounding only
    tol = 1e-12 if precision == 0 else 1e-4
    assert np.abs(xa - xb).max() < tol and np.abs(va - vb).max() < tol * np.sqrt(np.mean(va * va)) * 100
