"""Closing kicks and estimators of the batch engine over every class of bead
count, ragged last tiles (atom counts that are no multiple of 8) and one
molecule: against a single-system split handle of the same inputs (whose
estimators are FP64 on the same FP32 state) and, OBABO, its closing bath."""
import numpy as np
import pytest

from paper_2602_13553_gb300 import inputs
from tests._gpu import coord_err, pimd  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("integrator", [0, 1])
@pytest.mark.parametrize("nmol,P", [(33, 8), (35, 16), (130, 32), (50, 64), (43, 128), (45, 12), (36, 5), (700, 16)])
def test_batch_against_handle(pimd, nmol, P, integrator):
    L = inputs.box_length(nmol)
    x0, mass = inputs.water_lattice_box(nmol, L, P, 7, jitter=0.02)
    kw = dict(T=300.0, dt=5e-4, ff=inputs.water_ff_for_box(L), box=(L, L, L), seed=5, integrator=integrator)
    g = pimd.Simulation(x0, mass, potential=pimd.POT_WATERLIKE, precision=pimd.PREC_SPLIT, **kw)
    b = pimd.Batch(3)
    small_L = inputs.box_length(32)
    xs, ms = inputs.water_box(32, small_L, 20, 1, jitter=0.02)
    b.add(xs, ms, T=200.0, dt=5e-4, nsteps=10, ff=inputs.water_ff_for_box(small_L), box=(small_L,) * 3, seed=9)
    slot = b.add(x0, mass, nsteps=10, **kw)
    for n in (1, 2):
        g.step(n)
        b.run(n)
    xg, vg, sg = g.get_state()
    xb, vb, sb = b.get_state(slot)
    assert sg == sb == 3
    # the same arithmetic up to the order of FP32 sums in forces and transforms
    # (a few 1e-7 of a force a step) and the deviates' approximations (1e-6)
    assert np.abs(xg - xb).max() < 1e-4
    assert np.abs(vg - vb).max() < 5e-3 * np.sqrt(np.mean(vg * vg))
    eb = b.estimators()[slot]
    # the estimators' sums from the batch's own state: a handle at that state,
    # whose forces are FP32 like the batch's
    h = pimd.Simulation(xb, mass, v0=vb, potential=pimd.POT_WATERLIKE, precision=pimd.PREC_SPLIT, **kw)
    eh = h.estimators()
    for k in ("K_mode", "S_mode", "U_bead"):
        assert coord_err(eb[k], eh[k]) < 1e-5, k
    for k in ("H", "K_CV", "T_ring"):
        assert abs(eb[k] - eh[k]) < 1e-5 * abs(eh[k]), k
    h.close()
    g.close()
    b.close()
