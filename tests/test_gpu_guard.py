"""Faces whose FP32 Newton iteration falls towards vacuum: the FP32 forms mark
them and solve them again in FP64.  A gas torn apart (two halves receding
faster than their sound speed, short of generating vacuum) puts such faces on
the planes between the halves, in every chunk shape, on a static and a moving
mesh, with and without the entropy switch: the fluxes stay at the oracle's to
the FP32 forms' tolerance, every face is counted once, and a second step (whose
marks must have been cleared) does the same."""
import numpy as np
import pytest

from harness import ics
from oracle import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def amm():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_0901_4107_gb300 import amm as A
    return A


def torn(n, speed):
    P = ics.contact_3d(n, v=(0.0, 0.0, 0.0))
    c = np.sqrt(P.gamma * P.pres / P.rho)
    P.vel[:, 0] = np.where(P.tess.points[:, 0] < 0.5, -1.0, 1.0) * speed * c
    return P


@pytest.mark.parametrize("motion,entropy", [("eulerian", False), ("eulerian", True), ("lagrangian", False)])
def test_marked_faces(amm, motion, entropy):
    P = torn(14, 2.6)     # vacuum would take 2 / (gamma - 1) = 3 sound speeds
    Q, M = P.conserved(), O.Mesh(P.tess)
    V, s = O.geometry(M)
    W = O.primitives(M, Q, V, P.gamma)
    dt = 0.02 * O.timestep(M, W, V, None, P.gamma, 0.3)[0]
    wm = None if motion == "eulerian" else W[:, 1:4]
    F, cnt, rc = O.fluxes(M, W, O.gradients(M, W, V, s), s, wm, P.gamma, dt)
    assert rc == 0
    AF = F * P.tess.area[:, None]
    for block in (128, 256):
        ctx = amm.create_from_mesh(P.tess, Q, P.gamma, precision="fp32", mesh_motion=motion, entropy=entropy)
        amm.amm_set_tuning(ctx, 4, 2, block, 0)
        for step in range(2):
            amm.amm_set_state(ctx, Q)
            amm.amm_reset_stats(ctx)
            amm.amm_step(ctx, dt)
            st = amm.amm_get_stats(ctx)
            assert st["guard_faces"] > 50 and st["newton_fail"] == 0
            assert st["faces"] == P.n_faces == sum(st["newton_hist"])
            assert st["newton_iters"] >= sum(k * h for k, h in enumerate(st["newton_hist"]))
            e = np.abs(amm.amm_get_face_flux(ctx) - AF) / np.abs(AF).max(axis=0)
            assert e.max() < 2e-4, e.max()      # the FP32 flux tolerance of the parity tests
        amm.amm_destroy(ctx)
