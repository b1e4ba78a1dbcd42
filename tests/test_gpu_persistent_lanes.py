"""The one-launch step and the kernel sequence give the same bits in the FP32 and
FP64 forms at every launch shape, the defaults of each size among them (they
change with the number of cells; a mesh above the FP32 form's line)."""
import numpy as np
import pytest

from harness import ics
from tests.test_gpu_parity import amm  # noqa: F401

pytestmark = pytest.mark.gpu


def both(amm, make, shape=None, steps=2):  # noqa: F811
    outs = []
    for persistent, graph in ((0, False), (1, False), (1, True)):
        ctx = make()
        t = amm.amm_get_tuning(ctx)
        g, u = shape or (t["grad_lanes"], t["update_lanes"])
        amm.amm_set_tuning(ctx, g, u, t["flux_block"], persistent)
        amm.amm_advance(ctx, 0.3, steps, use_graph=graph)
        outs.append(amm.amm_get_state(ctx))
        amm.amm_destroy(ctx)
    assert np.array_equal(outs[0], outs[1]) and np.array_equal(outs[0], outs[2])
    return g, u


@pytest.mark.parametrize("entropy", [False, True])
@pytest.mark.parametrize("motion", ["eulerian", "lagrangian"])
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_every_shape(amm, prec, motion, entropy):  # noqa: F811
    P = ics.turbulent_3d(11, seed=2, mach=1.0)
    Q = P.conserved()
    for shape in (None, (1, 1), (2, 8), (8, 2), (4, 4), (1, 4)):
        both(amm, lambda: amm.create_from_mesh(P.tess, Q, P.gamma, precision=prec, mesh_motion=motion,
                                               entropy=entropy), shape)


def test_every_shape_of_an_ensemble(amm):  # noqa: F811
    E = ics.concat([ics.turbulent_3d(n, seed=n, mach=0.8) for n in (5, 7, 6)])
    for prec in ("fp32", "fp64"):
        for shape in (None, (2, 2), (8, 8)):
            both(amm, lambda: amm.amm_create(3, E.points, E.cells, E.shift, E.area, E.centroid, E.box, E.Q, E.gamma,
                                             amm.amm_default_options(prec, "eulerian"), box_cells=E.box_cells,
                                             box_faces=E.box_faces), shape)


@pytest.mark.parametrize("prec,n,lanes", [("fp32", 68, (2, 2)), ("fp64", 24, (2, 2)), ("fp64", 30, (1, 2))])
def test_defaults_above_the_lines(amm, prec, n, lanes):  # noqa: F811
    P = ics.turbulent_3d(n, seed=5)
    Q = P.conserved()
    assert both(amm, lambda: amm.create_from_mesh(P.tess, Q, P.gamma, precision=prec), steps=1) == lanes
