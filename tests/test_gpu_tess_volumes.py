"""The volumes of a tessellation fill the box without bias: their sum differs from it
by the mean of the cells' relative errors (2e-16 each at random), 2e-16 / sqrt(13824) =
2e-18 on a jittered lattice of 24^3, three of which are allowed besides the roundings of
the generators' own distances; a rounded 1/3 in place of the division alone is 5.6e-17."""
import numpy as np
import pytest

from harness import ics
from tests.test_gpu_voronoi import amm, gpu_tess  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seed", [1, 2, 3])
def test_volumes_are_not_biased(amm, seed):  # noqa: F811
    pts = ics.jittered_lattice((24,) * 3, np.ones(3), 0.4, np.random.default_rng(seed))
    vol = gpu_tess(amm, pts, np.ones(3))[1][4]
    assert abs(float(vol.astype(np.longdouble).sum() - 1)) < 1.5e-17
