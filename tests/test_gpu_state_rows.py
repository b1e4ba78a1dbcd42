"""The state and the primitives come back in the caller's order, whatever the
library's own order of the cells: less than a CTA's rows, ragged and whole tiles,
rows of four and of five words.  The state is returned bit for bit; the FP64
primitives to 1e-12 of their terms (the library sums its own volumes)."""
import numpy as np
import pytest

from harness import ics
from harness.tess import tessellate
from tests.test_gpu_update_lanes import amm  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(5, 5), (16, 16), (31, 17), (4, 4, 4), (8, 8, 8), (9, 8, 11)])
def test_rows(amm, shape):  # noqa: F811
    rng = np.random.default_rng(7)
    box = np.ones(len(shape))
    T = tessellate(ics.jittered_lattice(shape, box, 0.2, rng), box)
    n, d, g = T.n_cells, len(shape), 1.4
    order = rng.permutation(n)
    m = T.volume * (1.0 + order / n)
    v = rng.normal(size=(n, d))
    Q = np.column_stack([m, m[:, None] * v, T.volume * (2.0 + order) + 0.5 * m * (v * v).sum(1)])
    ctx = amm.create_from_mesh(T, Q, g, precision="fp64", mesh_motion="eulerian")
    assert np.array_equal(amm.amm_get_state(ctx), Q)
    Q2 = Q * 1.5
    amm.amm_set_state(ctx, Q2)
    assert np.array_equal(amm.amm_get_state(ctx), Q2)
    W = amm.amm_get_primitives(ctx)
    rho = Q2[:, 0] / T.volume
    u = Q2[:, 1:d + 1] / Q2[:, :1]
    e = Q2[:, -1] / T.volume
    want = np.column_stack([rho, u, (g - 1) * (e - 0.5 * rho * (u * u).sum(1))])
    scale = np.column_stack([rho, np.abs(u), (g - 1) * e])
    assert np.all(np.abs(W - want) <= 1e-12 * scale)        # (the volumes are the library's own sums)
    amm.amm_destroy(ctx)
