"""The FP64 water force (fixed-point Lennard-Jones pairs, one warp or several
per molecule and bead chunk) against the oracle: bead counts at the edges of the
chunks and lane groups, system sizes on both sides of every split, cutoffs far
beyond sigma (the scaled format), pairs closer than the fixed-point range,
scales that do not fit it, list rebuilds, unwrapped positions far from the box.

Positions and velocities after a few steps: the two sides differ by FP64
rounding, some 1e-14 of the largest force a step (stiff bonds); 1e-10 is the bar
of the harmonic tests, with steps to spare."""
import numpy as np
import pytest

from paper_2602_13553_gb300 import inputs
from tests._gpu import coord_err, pimd  # noqa: F401
from tests.test_gpu_parity import _pair

pytestmark = pytest.mark.gpu


def check(orc, pimd, x0, mass, L, ff, steps, **kw):
    c, g = _pair(orc, pimd, x0, mass, potential=1, ff=ff, box=(L, L, L), T=kw.pop("T", 300.0),
                 dt=kw.pop("dt", 5e-4), **kw)
    c.run(steps)
    g.step(steps)
    x, v, _ = g.get_state()
    assert coord_err(x, c.x) < 1e-10 and coord_err(v, c.v) < 1e-10
    eg, ec = g.estimators(), c.estimators()
    assert coord_err(eg["U_bead"], ec["U_bead"]) < 1e-10
    assert abs(eg["vir_sum"] - np.sum(c.vir)) < 1e-10 * (abs(np.sum(c.vir)) + abs(ec["H"]))
    g.close()


@pytest.mark.parametrize("nmol,P", [(24, 1), (33, 3), (200, 5), (70, 17), (64, 32), (130, 33), (90, 128), (300, 32),
                                    (520, 40), (530, 64)])
def test_sizes(orc, pimd, nmol, P):
    L = inputs.box_length(nmol)
    x0, mass = inputs.water_lattice_box(nmol, L, P, nmol + P, jitter=0.02)
    check(orc, pimd, x0, mass, L, inputs.water_ff_for_box(L), 4)


def test_images(orc, pimd):
    """Molecules left up to 40 boxes away: the forces of the starting positions
    through the energies, the virial and K_CV (no step, whose transforms would
    round at the size of the coordinates).  Separations carry 2 ulp(512 A) =
    2.3e-13 A against bond stretches of ~0.03 A: 1e-11 a bond, 1e-9 the bar."""
    L = inputs.box_length(64)
    x0, mass = inputs.water_lattice_box(64, L, 12, 3, jitter=0.02)
    x0 = x0 + L * np.repeat(np.random.default_rng(1).integers(-40, 40, size=(64, 3)), 3, axis=0)[None]
    c, g = _pair(orc, pimd, x0, mass, potential=1, ff=inputs.water_ff_for_box(L), box=(L, L, L), T=300.0, dt=5e-4)
    eg, ec = g.estimators(), c.estimators()
    assert coord_err(eg["U_bead"], ec["U_bead"]) < 1e-9
    assert abs(eg["vir_sum"] - np.sum(c.vir)) < 1e-9 * abs(np.sum(c.vir))
    assert abs(eg["K_CV"] - ec["K_CV"]) < 1e-9 * abs(ec["K_CV"])


@pytest.mark.parametrize("sig,rc", [(1.0, 6.0), (3.166, 9.0), (0.05, 4.0), (8.0, 4.0), (3.166, 3.3), (3.0, 0.005)])
def test_scales(orc, pimd, sig, rc):
    L = 20.0
    x0, mass = inputs.water_lattice_box(70, L, 8, 5, jitter=0.02)
    ff = list(inputs.WATER_FF)
    ff[4], ff[5], ff[6] = (1e-9 if sig > 4 else 6.7e-3), sig, rc
    check(orc, pimd, x0, mass, L, tuple(ff), 3)


@pytest.mark.parametrize("gap", [0.9, 1.9, 2.0, 2.05])
def test_close_pairs(orc, pimd, gap):
    """Oxygens closer than the fixed-point range (2 A here) and next to it."""
    L = inputs.box_length(40)
    x0, mass = inputs.water_lattice_box(40, L, 6, 9, jitter=0.02)
    shift = x0[:, 0:1] + np.array([gap, 0.0, 0.0]) - x0[:, 3:4]
    x0[:, 3:6] += shift
    check(orc, pimd, x0, mass, L, inputs.water_ff_for_box(L), 2, dt=1e-5)


@pytest.mark.parametrize("nmol,P", [(64, 8), (540, 64)])
def test_rebuilds(orc, pimd, nmol, P):
    """Two half boxes sheared past each other at +-100 A/ps for 20 fs: the lists
    are rebuilt on the way, and pairs meet that started beyond cutoff and skin.
    The water bar of the parity tests, 1e-8."""
    L = inputs.box_length(nmol)
    x0, mass = inputs.water_lattice_box(nmol, L, P, 4, jitter=0.02)
    up = np.repeat(x0[0, 0::3, 2] < 0.5 * L, 3)
    v0 = np.zeros_like(x0)
    v0[0, :, 1] = np.where(up, 100.0, -100.0) * np.sqrt(P)
    c, g = _pair(orc, pimd, x0, mass, v0=v0, potential=1, ff=inputs.water_ff_for_box(L), box=(L, L, L), T=300.0,
                 dt=5e-4)
    c.run(40)
    g.step(40)
    x, v, _ = g.get_state()
    assert 2.0 * np.abs(x[:, 0::3].mean(0) - x0[:, 0::3].mean(0)).max() > 1.5
    assert coord_err(x, c.x) < 1e-8 and coord_err(v, c.v) < 1e-8
    g.close()


@pytest.mark.parametrize("nmol,P", [(160, 32), (610, 64)])
def test_warps_per_unit(orc, pimd, nmol, P):
    """Units of 7 list warps, and one-warp units with the list check apart, over
    rebuilds of the lists (the bar of test_rebuilds)."""
    test_rebuilds(orc, pimd, nmol, P)
