"""Individual time steps where the signal-speed walk, the few-face flux form and
the few-cell gradients change their path, against the oracle's cycle: buckets
of very uneven filling (a scan in several parts, empty buckets), two pyramid
levels (the smallest tree), neighbouring faces of strongly different states
(shocks, rarefactions and generated vacuum in the lanes of one warp), more and
fewer active faces and cells than the small-tick forms take.  Bins and counters
are equal; the states agree to 1e-12 per element (sums of some 15 fluxes in
another order, 2^-52 each, through at most a few hundred sub-steps)."""
import numpy as np
import pytest

from harness import ics
from harness.tess import tessellate
from oracle import oracle as O
from tests.test_gpu_individual import amm, rel_err  # noqa: F401

pytestmark = pytest.mark.gpu


def uneven(shape, power, seed):
    """A jittered lattice drawn towards the origin: u -> u^power per axis."""
    rng = np.random.default_rng(seed)
    box = np.ones(len(shape))
    u = np.mod(ics.jittered_lattice(shape, box, 0.3, rng), 1.0)
    return tessellate(u ** power, box), rng


@pytest.mark.parametrize("shape,power,contrast,mach,dt", [
    ((4, 4, 4), 1.0, 2.0, 0.5, 2e-2),        # two levels
    ((14, 14, 14), 3.0, 0.7, 0.2, 2e-4),     # 343 cells in one bucket, most buckets with none or one
    ((7, 9), 1.0, 2.0, 0.5, 2e-2),
    ((40, 40), 2.0, 2.0, 0.5, 1e-3),
    ((12, 12, 12), 1.0, 2.0, 6.0, 1e-4),     # generated vacuum beside shocks
    ((24, 24, 24), 1.0, 0.7, 0.2, 4e-3),     # more active faces than the small form takes
])
def test_uneven_states_match_oracle(amm, shape, power, contrast, mach, dt):  # noqa: F811
    T, rng = uneven(shape, power, 11 + len(shape))
    M = O.Mesh(T)
    V, s = O.geometry(M)
    g, d = 5.0 / 3.0, len(shape)
    rho = 10.0 ** rng.uniform(-0.5 * contrast, 0.5 * contrast, len(V))
    P = 10.0 ** rng.uniform(-contrast, contrast, len(V))
    v = mach * np.sqrt(g * P / rho)[:, None] * rng.uniform(-1.0, 1.0, (len(V), d))
    m = V * rho
    Q = np.column_stack([m, m[:, None] * v, V * P / (g - 1) + 0.5 * m * (v * v).sum(1)])
    Qo, bo, co, rc = O.advance_individual(M, Q.copy(), g, 0.3, dt, max_depth=30, signal=True, geom=(V, s))
    assert rc == 0
    ctx = amm.create_from_mesh(T, Q, g, precision="fp64", mesh_motion="eulerian")
    st = amm.amm_advance_individual(ctx, 0.3, dt, 30, True)
    Qg, bg = amm.amm_get_state(ctx), amm.amm_get_bins(ctx)
    amm.amm_destroy(ctx)
    assert np.array_equal(bo, bg)
    assert (st["substeps"], st["face_fluxes"], st["activations"]) == (co[4], co[5], co[6])
    assert rel_err(Qg, Qo, Q, M, V, g) < 1e-12
