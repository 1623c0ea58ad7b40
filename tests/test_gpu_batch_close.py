"""The closing kick of the batch's warp items: F~ = M F in FP32.

Molecules start at the exact rest geometry, out of one another's reach, all beads
in one place and moving as one: the opening kick and every transform before the
closing kick are exact zeros in the internal modes, and the forces of the new
positions are the same in every bead.  What the internal modes' velocities hold
after one step is the error of that transform alone, in units of the centroid
mode's kick."""
import numpy as np
import pytest

from tests._gpu import pimd  # noqa: F401

pytestmark = pytest.mark.gpu


def fma(a, b, c):
    return np.float32(np.float64(a) * np.float64(b) + np.float64(c))


def mode_matrix(P):
    j = np.arange(P)
    M = np.empty((P, P))
    for k in range(P):
        if k == 0:
            M[k] = 1.0
        elif 2 * k == P:
            M[k] = (-1.0) ** j
        else:
            M[k] = np.sqrt(2.0) * (np.cos if 2 * k < P else np.sin)(2 * np.pi * ((k * j) % P) / P)
    return M / np.sqrt(P)


@pytest.mark.parametrize("P", [8, 16, 32, 64, 128])
def test_closing_kick_error(pimd, P):
    """No further off than the FP32 sum over a whole row in two chains, terms in
    order (emulated here on the same forces, rounding by rounding)."""
    rng = np.random.default_rng(P)
    k = 3
    nmol = k ** 3
    L = 8.0 * k
    site = 8.0 * np.stack(np.meshgrid(*[np.arange(k)] * 3, indexing="ij"), -1).reshape(-1, 3) + 2.0
    x = np.empty((1, 3 * nmol, 3))
    x[0, 0::3] = site
    x[0, 1::3] = site + np.array([1.0, 0.0, 0.0])
    x[0, 2::3] = site + np.array([0.0, 1.0, 0.0])
    x = np.repeat(x, P, axis=0)
    v0 = np.zeros_like(x)
    v0[0] = rng.normal(0.0, 100.0, x.shape[1:])
    mass = np.tile([15.999, 1.008, 1.008], nmol)
    dt = 1e-3
    b = pimd.Batch(1)
    s = b.add(x, mass, v0=v0, T=300.0, dt=dt, nsteps=1, ff=(40.0, 1.0, 5.0, np.pi / 2, 6.7e-3, 3.0, 3.9, 0.0),
              box=(L,) * 3, seed=1, thermostat=0)
    b.run(1)
    _, v, _ = b.get_state(s)
    b.close()
    kick = v[0] - v0[0]                      # (h / 2m) sqrt(P) F
    on = np.abs(kick) > 0.1 * np.abs(kick).max()
    assert on.sum() > nmol
    err = (v[1:] / kick)[:, on]
    # the same quotient for the plain FP32 sum of P equal forces
    M = mode_matrix(P).astype(np.float32)
    F = np.float32(kick[on] * mass.repeat(3).reshape(-1, 3)[on])
    ref = np.empty((P - 1, F.size))
    for q in range(1, P):
        fa, fb = np.zeros(F.size, np.float32), np.zeros(F.size, np.float32)
        for j in range(0, P, 2):
            fa, fb = fma(M[q, j], F, fa), fma(M[q, j + 1], F, fb)
        ref[q - 1] = (fa + fb) / (np.sqrt(P) * F.astype(float))
    rms, bar = np.sqrt(np.mean(err ** 2)), np.sqrt(np.mean(ref ** 2))
    print("P = %d: closing kick rms %.2e, plain FP32 sum %.2e" % (P, rms, bar))
    assert rms <= 1.1 * bar
