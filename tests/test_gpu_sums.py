"""fixcom and the barostat's kick as reductions over all atoms, against the
oracle: bead counts at the edges of the lane groups (1, 2, 3, 33, 40, 128),
one atom, more atoms than one round of groups, both methods and integrators,
and fixcom together with the barostat.  Bars as in the method tests: 1e-10
(harmonic), 1e-8 (water-like)."""
import math

import numpy as np
import pytest

from paper_2602_13553_gb300 import inputs
from tests._gpu import coord_err, pimd  # noqa: F401
from tests.test_gpu_parity import _pair

pytestmark = pytest.mark.gpu

OMEGA_HO = 0.1 / (4.135667403e-3 / (2 * math.pi))


@pytest.mark.parametrize("method,integrator,N,P", [(0, 0, 1, 1), (0, 1, 500, 3), (0, 1, 50, 40), (0, 0, 3000, 16),
                                                   (1, 0, 40, 33), (1, 1, 30, 128), (1, 0, 700, 2), (1, 1, 9, 1)])
def test_fixcom_sizes(orc, pimd, method, integrator, N, P):
    x0, mass = inputs.harmonic(N, P, seed=N + P, std=0.1)
    mass = mass * (1.0 + np.arange(N) % 3)
    c, g = _pair(orc, pimd, x0, mass, T=300.0, dt=2.5e-4, potential=0, ff=(OMEGA_HO,), integrator=integrator,
                 method=method, fixcom=1)
    c.run(6)
    g.step(2)
    g.step(4)
    x, v, _ = g.get_state()
    assert coord_err(x, c.x) < 1e-10
    assert np.max(np.abs(v - c.v)) < 1e-10 * max(1.0, float(np.sqrt(np.mean(c.v * c.v))))


@pytest.mark.parametrize("barostat,integrator,P,fixcom", [(1, 0, 1, 0), (2, 1, 33, 0), (1, 1, 3, 1), (2, 0, 20, 1)])
def test_barostat_sizes(orc, pimd, barostat, integrator, P, fixcom):
    L = inputs.box_length(40)
    x0, mass = inputs.water_box(40, L, P, 5, jitter=0.02)
    c, g = _pair(orc, pimd, x0, mass, T=300.0, dt=2.5e-4, potential=1, ff=inputs.water_ff_for_box(L),
                 box=(L, L, L), integrator=integrator, barostat=barostat, pext=5e-3, taup=0.1, fixcom=fixcom)
    c.run(10)
    g.step(10)
    x, v, _ = g.get_state()
    assert coord_err(x, c.x) < 1e-8 and coord_err(v, c.v) < 1e-8
    vw, box = g.get_barostat()
    want = c.vW if barostat == 1 else np.array(list(c.vWa))
    assert np.max(np.abs(vw - want)) < 1e-8 * max(1.0, float(np.max(np.abs(want))))
    assert np.abs(box - c.box).max() < 1e-10 * c.box.max()
