"""The update kernel's lanes per cell: the FP32 forms' flux sums are exact
integers, so the state after a step is the same bit for bit however a cell's
incidences are split over lanes, and the FP64 form's agrees to the rounding of
its sums.  Sizes: less than one warp's cells, a tile's edge, ragged tiles,
several boxes, and a cell with more faces than one run of 32-bit digit sums
holds.  The totals are the sums of the state."""
from dataclasses import replace

import numpy as np
import pytest

from harness import ics
from oracle import oracle as O

pytestmark = pytest.mark.gpu
EPS = np.finfo(np.float64).eps


@pytest.fixture(scope="module")
def amm():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_0901_4107_gb300 import amm as A
    return A


def pieces(k=60):
    """A 2D box whose cell 0 has each of its faces cut into k collinear pieces
    (cells that close are all the update asks of a mesh)."""
    P = ics.gresho_2d(9, jitter=0.1)
    T = P.tess
    cut = np.any(T.cells == 0, axis=1)
    at = np.repeat(np.arange(T.n_faces), np.where(cut, k, 1))
    part = np.concatenate([np.arange(k if c else 1) for c in cut])
    d = T.points[T.cells[:, 1]] + T.shift * T.box - T.points[T.cells[:, 0]]
    along = np.column_stack([-d[:, 1], d[:, 0]]) / np.linalg.norm(d, axis=1)[:, None]
    n = np.where(cut, k, 1)[at]
    off = ((part + 0.5) / n - 0.5) * T.area[at]
    T = replace(T, cells=T.cells[at].copy(), shift=T.shift[at].copy(), area=T.area[at] / n,
                centroid=T.centroid[at] + off[:, None] * along[at],
                faces_per_cell=np.bincount(T.cells[at].ravel(), minlength=T.n_cells))
    return replace(P, tess=T)


PROBLEMS = {"few": lambda: ics.turbulent_3d(4, seed=1, mach=0.5), "tile": lambda: ics.gresho_2d(16, jitter=0.1),
            "ragged": lambda: ics.turbulent_3d(11, seed=2, mach=1.0), "pieces": pieces}


@pytest.mark.parametrize("entropy", [False, True])
@pytest.mark.parametrize("name", sorted(PROBLEMS))
def test_lanes_do_not_change_the_step(amm, name, entropy):
    P = PROBLEMS[name]()
    Q = P.conserved()
    if name == "pieces":
        assert P.tess.faces_per_cell.max() > 256
    dt = O.step(O.Mesh(P.tess), Q, P.gamma, "lagrangian", cfl=0.3)[1]
    for prec in ("fp32", "fp64"):
        outs = []
        for lanes in (1, 2, 4, 8):
            ctx = amm.create_from_mesh(P.tess, Q, P.gamma, precision=prec, entropy=entropy)
            amm.amm_set_tuning(ctx, 4, lanes, 256, 0)
            amm.amm_step(ctx, dt)
            outs.append(amm.amm_get_state(ctx))
            tot = amm.amm_get_totals(ctx)[0]
            assert np.all(np.abs(tot - outs[-1].sum(0)) <= len(Q) * EPS * np.abs(outs[-1]).sum(0))
            flux = amm.amm_get_face_flux(ctx)
        if prec == "fp32":
            for o in outs[1:]:
                assert np.array_equal(o, outs[0])
        else:
            # a cell's sum of m terms in two orders: m eps sum |dt A F| each,
            # m the largest number of faces; the state's own rounding
            m = P.tess.faces_per_cell.max()
            mag = np.zeros_like(Q)
            np.add.at(mag, P.tess.cells[:, 0], np.abs(flux))
            np.add.at(mag, P.tess.cells[:, 1], np.abs(flux))
            for o in outs[1:]:
                bound = 2 * m * EPS * dt * mag + 4 * EPS * np.abs(o)
                if entropy:   # (an energy from the entropy repeats it through rho^gamma)
                    bound[:, -1] += 32 * m * EPS * np.abs(o[:, -1])
                assert np.all(np.abs(o - outs[0]) <= bound)


def test_lanes_in_an_ensemble(amm):
    E = ics.concat([ics.turbulent_3d(n, seed=n, mach=0.8) for n in (5, 7, 6)])
    outs = []
    for lanes in (1, 2, 4, 8):
        ctx = amm.amm_create(3, E.points, E.cells, E.shift, E.area, E.centroid, E.box, E.Q, E.gamma,
                             amm.amm_default_options("fp32", "eulerian"), box_cells=E.box_cells,
                             box_faces=E.box_faces)
        amm.amm_set_tuning(ctx, 2, lanes, 256, 0)
        amm.amm_advance(ctx, 0.3, 2)
        outs.append((amm.amm_get_state(ctx), amm.amm_get_totals(ctx)))
    for q, t in outs:
        assert np.array_equal(q, outs[0][0])
        for b in range(3):
            s = q[E.box_cells[b]:E.box_cells[b + 1]]
            assert np.all(np.abs(t[b] - s.sum(0)) <= len(s) * EPS * np.abs(s).sum(0))
