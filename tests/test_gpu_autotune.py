"""The autotuner's search over the blocks per SM of the 64-bead step kernel."""
import pytest

from paper_2602_13553_gb300 import inputs
from tests._gpu import pimd  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("trial", [1, 5])
def test_every_grid_is_tried(pimd, trial):
    """One settling step, then two trials of every grid from one block an SM to the
    four that the kernel's registers let on it."""
    b = pimd.Batch(2)
    slots = []
    for nmol, seed in ((32, 1), (40, 2)):
        L = inputs.box_length(nmol)
        x0, mass = inputs.water_box(nmol, L, 64, seed, jitter=0.02)
        slots.append(b.add(x0, mass, T=300.0, dt=5e-4, nsteps=1000, ff=inputs.water_ff_for_box(L), box=(L,) * 3,
                           seed=seed))
    tiles = b.autotune(trial)
    st, _ = b.status()
    assert all(int(st[s]) == 1 + 2 * 4 * trial for s in slots)
    assert 1 <= tiles["warp_blocks_per_sm"] <= 4
    b.close()
