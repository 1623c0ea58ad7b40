"""Checkpoint and resume through get_state and set_state: bit for bit in FP64 (the
lists are rebuilt on the way in, the positions wrapped anew)."""
import numpy as np
import pytest

from paper_2602_13553_gb300 import inputs
from tests._gpu import pimd  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("integ", [0, 1])
@pytest.mark.parametrize("nmol,P", [(64, 16), (300, 64)])
def test_fp64_resume_is_bitwise(pimd, nmol, P, integ):
    L = inputs.box_length(nmol)
    x0, mass = inputs.water_lattice_box(nmol, L, P, 3, jitter=0.02)
    x0 = x0 + L * np.repeat(np.random.default_rng(1).integers(-3, 4, size=(nmol, 3)), 3, axis=0)[None]
    kw = dict(T=300.0, dt=5e-4, potential=1, ff=inputs.water_ff_for_box(L), box=(L,) * 3, seed=11, integrator=integ)
    a = pimd.Simulation(x0, mass, **kw)
    a.step(25)
    x, v, st = a.get_state()
    a.step(15)
    b = pimd.Simulation(x0, mass, **kw)
    b.set_state(x, v, st)
    b.step(15)
    for p, q in zip(a.get_state(), b.get_state()):
        assert np.array_equal(p, q)
