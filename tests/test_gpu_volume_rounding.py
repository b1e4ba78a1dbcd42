"""Cell volumes (Sec. 3, V = sum of the pyramids A h / dim): the roundings are
unbiased, so over thousands of cells the mean relative error against long double is
far below a single one (an ulp is 2.2e-16, the mean of 13824 cells' errors of about
1e-16 each some 1e-18; a rounded 1/3 in place of the division alone is 5.6e-17)."""
import numpy as np
import pytest

from harness import ics
from tests.test_gpu_parity import amm  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim", [2, 3])
def test_volumes_are_not_biased(amm, dim):  # noqa: F811
    P = ics.turbulent_3d(24, seed=3) if dim == 3 else ics.gresho_2d(100, jitter=0.3)
    T = P.tess
    x, b = T.points.astype(np.longdouble), np.asarray(T.box, np.longdouble)
    d = x[T.cells[:, 1]] + T.shift * b - x[T.cells[:, 0]]
    vp = T.area.astype(np.longdouble) * (np.sqrt((d * d).sum(1)) / 2) / dim
    V = np.zeros(T.n_cells, np.longdouble)
    np.add.at(V, T.cells[:, 0], vp)
    np.add.at(V, T.cells[:, 1], vp)
    ctx = amm.create_from_mesh(T, P.conserved(), P.gamma, precision="fp64")
    e = ((amm.amm_get_geometry(ctx)[0] - V) / V).astype(np.float64)
    print(dim, e.mean(), e.std())
    assert e.std() < 3e-16 and abs(e.mean()) < 1.5e-17
