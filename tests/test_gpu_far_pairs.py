"""The FP64 water force where every O-O pair is near the cutoff: a lattice of
spacing 0.9 rc, all coordinates multiples of 2^-20 A (separations are exact on
both sides), bonds and angles switched off, so that energy, virial and forces are
sums of the smallest pair terms alone."""
import numpy as np
import pytest

from tests._gpu import coord_err, pimd  # noqa: F401
from tests.test_gpu_parity import _pair

pytestmark = pytest.mark.gpu


def far_lattice(k, rc, P, seed):
    rng = np.random.default_rng(seed)
    q = 2.0 ** -20
    a = np.rint(0.9 * rc * 1024) / 1024
    site = a * np.stack(np.meshgrid(*[np.arange(k)] * 3, indexing="ij"), -1).reshape(-1, 3)
    O = site[None] + np.rint(rng.uniform(-0.03, 0.03, (1, k ** 3, 3)) * rc / q) * q
    O = O + np.rint(rng.uniform(-0.01, 0.01, (P, k ** 3, 3)) * rc / q) * q
    x = np.empty((P, 3 * k ** 3, 3))
    x[:, 0::3] = O
    x[:, 1::3] = O + np.array([0.75, 0.5, 0.0])
    x[:, 2::3] = O + np.array([-0.75, 0.5, 0.0])
    return x, np.tile([15.999, 1.008, 1.008], k ** 3), k * a


@pytest.mark.parametrize("sig,rc", [(3.166, 7.9), (3.166, 12.0), (3.166, 20.0), (1.0, 7.9), (0.5, 3.9)])
@pytest.mark.parametrize("k,P", [(4, 1), (4, 9), (6, 64), (9, 64)])
def test_far_pairs(orc, pimd, k, P, sig, rc):
    """A pair carries some 1e-15 of its own size on either side; sums of up to
    2e5 like-signed terms in FP64 (the oracle's) add sqrt(n) 1e-16: 5e-14."""
    x, mass, L = far_lattice(k, rc, P, 7 * k + P)
    ff = (0.0, 1.0, 0.0, 1.824, 6.7e-3, sig, rc, 0.0)
    c, g = _pair(orc, pimd, x, mass, v0=np.zeros_like(x), potential=1, ff=ff, box=(L, L, L), T=300.0, dt=1e-4,
                 thermostat=0)
    eg, ec = g.estimators(), c.estimators()
    assert coord_err(eg["U_bead"], ec["U_bead"]) < 5e-14
    assert abs(eg["vir_sum"] - np.sum(c.vir)) < 5e-14 * abs(np.sum(c.vir))
    if P == 1:   # forces: the velocities of one step from rest
        c.run(1)
        g.step(1)
        _, v, _ = g.get_state()
        assert coord_err(v[:, 0::3], c.v[:, 0::3]) < 5e-14
    g.close()
