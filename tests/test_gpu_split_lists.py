"""Split-precision water forces depend on the interacting pairs, not on what else
the neighbour list holds: a molecule between the cutoff and the list's radius,
which interacts with nothing, changes no bit of the others' motion."""
import numpy as np
import pytest

from paper_2602_13553_gb300 import inputs
from tests._gpu import pimd  # noqa: F401

pytestmark = pytest.mark.gpu

# molecules and beads on every split of a unit's list (7 warps, 2, 1), with one
# and with many molecules a warp
SIZES = [(40, 64), (150, 5), (36, 3), (520, 33), (700, 64)]


@pytest.mark.parametrize("nmol,P", SIZES)
def test_idle_candidates_change_nothing(pimd, nmol, P):
    rc = 6.0
    L = inputs.box_length(nmol)
    x0, mass = inputs.water_lattice_box(nmol, L, P, nmol, jitter=0.02)
    x0 = x0 - x0[:, 0::3].mean(0).mean(0)
    big = L + 24.0   # no images within reach
    # rings of idle molecules 6.6 A beyond the faces of the cluster, 6.6 A or more
    # apart from each other: inside rc + skin = 7.5 A of the outer molecules
    O = x0[:, 0::3].mean(0)
    idle = []
    for axis in range(3):
        for sign in (-1.0, 1.0):
            for t in (np.array([-0.3, -0.3]), np.array([0.3, 0.3]), np.array([-0.3, 0.3])):
                p = np.zeros(3)
                p[[a for a in range(3) if a != axis]] = t * L
                p[axis] = sign * (L + 20.0) / 2
                # pull it in along the axis until its nearest oxygen is 6.6 A away
                while True:
                    q = p.copy()
                    q[axis] -= sign * 0.01
                    if np.linalg.norm(O - q, axis=1).min() < 6.6:
                        break
                    p = q
                if all(np.linalg.norm(p - o) > 6.6 for o in idle):
                    idle.append(p)
    assert len(idle) >= 6
    geo = x0[:, 0:3] - x0[:, 0:1]
    assert all(np.linalg.norm(x0[:, 0::3] - p, axis=2).min() > rc + 0.2 for p in idle)
    shell = sum(int((np.linalg.norm(O - p, axis=1) < 7.5).sum()) for p in idle)
    assert shell >= len(idle)
    extra = np.concatenate([geo + p for p in idle], axis=1)
    out = []
    for x, m in ((x0, mass), (np.concatenate([x0, extra], 1), np.concatenate([mass, np.tile(mass[:3], len(idle))]))):
        g = pimd.Simulation(x, m, v0=np.zeros_like(x), T=100.0, dt=2e-4, potential=1, ff=inputs.WATER_FF,
                            box=(big,) * 3, seed=5, precision=pimd.PREC_SPLIT)
        g.step(3)
        xs, vs, _ = g.get_state()
        out.append((xs[:, :3 * nmol], vs[:, :3 * nmol]))
        g.close()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])


def test_energy_sums_do_not_depend_on_the_split(pimd):
    """U and Tr Xi of one cluster of 64 molecules, its units' lists shared by seven
    warps, by two and taken by one (idle molecules out of every reach bring the
    number of units there; bonds and angles off): the FP32 terms are the same ones,
    and sums that keep their rounding errors lose 2^-48 an addition, 190 additions
    at most: 1e-12 of the terms' magnitudes, 1e-11 where they cancel by ten."""
    P, L = 64, 12.42
    x0, mass = inputs.water_lattice_box(64, L, P, 2, jitter=0.02)
    x0 = x0 - x0[:, 0::3].mean(0).min(0)   # the cluster in a corner
    big, a = 96.0, 8.0
    g = np.stack(np.meshgrid(*[np.arange(2, 12) * a - 4.0] * 3, indexing="ij"), -1).reshape(-1, 3)
    site = g[np.linalg.norm(np.maximum(g - L, 0.0), axis=1) > 7.9]
    ff = (0.0,) + inputs.WATER_FF[1:2] + (0.0,) + inputs.WATER_FF[3:]
    geo = x0[:1, 0:3] - x0[:1, 0:1]
    out = []
    for idle in (0, 236, 600):
        x = np.concatenate([x0] + [np.repeat(geo + p, P, axis=0) for p in site[:idle]], axis=1)
        sim = pimd.Simulation(x, np.tile(mass[:3], x.shape[1] // 3), v0=np.zeros_like(x), T=300.0, dt=1e-4,
                              potential=1, ff=ff, box=(big,) * 3, seed=5, precision=pimd.PREC_SPLIT)
        e = sim.estimators()
        out.append((e["U_bead"], e["vir_sum"]))
        sim.close()
    for u, w in out[1:]:
        assert np.abs(u - out[0][0]).max() < 1e-11 * np.abs(out[0][0]).max()
        assert abs(w - out[0][1]) < 1e-11 * abs(out[0][1])
