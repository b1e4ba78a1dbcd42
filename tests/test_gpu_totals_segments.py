"""A box's totals when its block partials are cut into segments (more than 2040
sums) and when not, for one box and for boxes of very different sizes that share a
launch (segments of a small box are then empty), after a step and without one.  The
totals are the state's sums to the rounding of n additions in some order: 2 eps
times the additions on one thread's chain (at most 64 here), of sum |Q|."""
import numpy as np
import pytest

from harness import ics
from tests.test_gpu_update_lanes import amm  # noqa: F401

pytestmark = pytest.mark.gpu


def check(amm, ctx, cells):  # noqa: F811
    Q, tot = amm.amm_get_state(ctx), amm.amm_get_totals(ctx)
    at = np.concatenate([[0], np.cumsum(cells)])
    for b in range(len(cells)):
        q = Q[at[b]:at[b + 1]]
        assert np.all(np.abs(tot[b] - q.sum(0)) <= 128 * np.finfo(float).eps * np.abs(q).sum(0)), b


@pytest.mark.parametrize("sizes,lanes", [([12], 8), ([38], 2), ([38], 8), ([38, 6, 12], 8)])
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_totals(amm, sizes, lanes, prec):  # noqa: F811
    Ps = [ics.turbulent_3d(n, seed=3 + k) for k, n in enumerate(sizes)]
    E = ics.concat(Ps)
    ctx = amm.amm_create(3, E.points, E.cells, E.shift, E.area, E.centroid, E.box, E.Q, E.gamma,
                         amm.amm_default_options(prec, "eulerian"), box_cells=E.box_cells, box_faces=E.box_faces)
    amm.amm_set_tuning(ctx, 4, lanes, 256, 0)
    cells = [P.tess.n_cells for P in Ps]
    check(amm, ctx, cells)
    for _ in range(2):
        amm.amm_advance(ctx, 0.3, 2)
        check(amm, ctx, cells)
    amm.amm_destroy(ctx)
