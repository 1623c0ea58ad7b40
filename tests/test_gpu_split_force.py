"""The split-precision water force of single systems against the oracle: bead
counts at the edges of the chunks and lane groups, list lengths odd and even,
system sizes on both sides of every split of a neighbour list, rebuilds.  Bars of
the split-precision path (tests/_gpu.py)."""
import numpy as np
import pytest

from paper_2602_13553_gb300 import inputs
from tests._gpu import assert_split_close, pimd  # noqa: F401
from tests.test_gpu_parity import _pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nmol,P,steps", [(24, 1, 6), (33, 3, 6), (71, 17, 6), (64, 32, 6), (130, 33, 6), (300, 64, 4),
                                          (700, 96, 3), (2100, 64, 2)])
def test_sizes(orc, pimd, nmol, P, steps):
    L = inputs.box_length(nmol)
    x0, mass = inputs.water_lattice_box(nmol, L, P, nmol + P, jitter=0.02)
    c = orc.Sim(x0, mass, T=300.0, dt=5e-4, potential=1, ff=inputs.water_ff_for_box(L), box=(L, L, L), seed=3)
    g = pimd.Simulation(x0, mass, T=300.0, dt=5e-4, potential=1, ff=inputs.water_ff_for_box(L), box=(L, L, L),
                        seed=3, precision=pimd.PREC_SPLIT)
    c.run(steps)
    g.step(steps)
    x, v, _ = g.get_state()
    assert_split_close(x, v, g.estimators(), c, c.estimators(), "%d x %d" % (nmol, P))
    g.close()


@pytest.mark.parametrize("nmol,P", [(64, 20), (530, 32), (1100, 128)])
def test_rebuilds(pimd, nmol, P):
    """Two half boxes sheared past each other, with the lists rebuilt on the way,
    against the FP64 handle on the same inputs.  Positions only: 1e-4 A, the bar
    of the split path (velocities of colliding molecules amplify FP32 rounding)."""
    L = inputs.box_length(nmol)
    x0, mass = inputs.water_lattice_box(nmol, L, P, 4, jitter=0.02)
    up = np.repeat(x0[0, 0::3, 2] < 0.5 * L, 3)
    v0 = np.zeros_like(x0)
    v0[0, :, 1] = np.where(up, 100.0, -100.0) * np.sqrt(P)
    out = []
    for prec in (pimd.PREC_FP64, pimd.PREC_SPLIT):
        g = pimd.Simulation(x0, mass, v0=v0, T=300.0, dt=5e-4, potential=1, ff=inputs.water_ff_for_box(L),
                            box=(L, L, L), seed=3, precision=prec)
        g.step(24)
        out.append(g.get_state()[0])
        g.close()
    assert 2.0 * np.abs(out[0][:, 0::3].mean(0) - x0[:, 0::3].mean(0)).max() > 1.5
    assert np.abs(out[0] - out[1]).max() < 1e-4
