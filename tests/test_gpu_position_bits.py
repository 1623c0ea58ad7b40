"""The FP64 water force in boxes on both sides of the edges where its positions change
format (53 fraction bits below 256 A, 50 below 2048 A, FP64 pairs from there on): a
liquid cluster around the origin, so that molecules sit at both ends of the box,
against the oracle at the bars of tests/test_gpu_force_fixed.py."""
import pytest

from paper_2602_13553_gb300 import inputs
from tests._gpu import pimd  # noqa: F401
from tests.test_gpu_force_fixed import check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [255.9, 256.0, 2047.0, 2048.0])
@pytest.mark.parametrize("nmol,P", [(70, 8), (230, 64), (620, 64)])
def test_boxes(orc, pimd, nmol, P, L):
    l = inputs.box_length(nmol)
    x0, mass = inputs.water_lattice_box(nmol, l, P, nmol, jitter=0.02)
    check(orc, pimd, x0 - 0.5 * l, mass, L, inputs.WATER_FF, 2)
