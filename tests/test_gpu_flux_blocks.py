"""The FP64 flux kernel's CTA sizes, on both sides of the number of faces up to
which 64 is the default: the setting is the one that runs, faces come out bit
for bit alike (a face's arithmetic does not depend on the CTA it is in, nor on
the grouping of the solves that 128 and 256 do), and a step has oracle parity
(1e-12, the FP64 form's)."""
import numpy as np
import pytest

from harness import ics
from oracle import oracle as O
from tests.test_gpu_parity import TOL, amm, errs, floor_of  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("entropy", [False, True])
@pytest.mark.parametrize("n,default", [(16, 64), (28, 256)])
def test_blocks_agree(amm, n, default, entropy):  # noqa: F811
    P = ics.turbulent_3d(n, seed=2)
    assert (P.tess.n_faces <= 152 * 1024) == (default == 64)
    M = O.Mesh(P.tess)
    Q = P.conserved()
    ref, dt, _, _ = O.step(M, Q, P.gamma, "lagrangian", cfl=0.3)
    fl = floor_of(Q, 3, P.gamma, O.primitives(M, Q, P.tess.volume, P.gamma))
    outs = []
    for block in (None, 64, 128, 256):
        ctx = amm.create_from_mesh(P.tess, Q, P.gamma, precision="fp64", entropy=entropy)
        t = amm.amm_get_tuning(ctx)
        if block is None:
            assert t["flux_block"] == default
        else:
            amm.amm_set_tuning(ctx, t["grad_lanes"], t["update_lanes"], block, 0)
            assert amm.amm_get_tuning(ctx)["flux_block"] == block
        amm.amm_step(ctx, dt)
        st = amm.amm_get_stats(ctx)
        outs.append((amm.amm_get_face_flux(ctx), amm.amm_get_state(ctx), st["newton_hist"], st["newton_iters"]))
        amm.amm_destroy(ctx)
    for o in outs[1:]:
        assert np.array_equal(o[0], outs[0][0]) and np.array_equal(o[1], outs[0][1]) and o[2:] == outs[0][2:]
    if not entropy:
        assert errs(outs[0][1], ref, fl)[0] < TOL["fp64"]


def test_sixty_four_is_of_the_fp64_form(amm):  # noqa: F811
    P = ics.turbulent_3d(8, seed=3)
    for prec in ("fp64", "fp32"):
        ctx = amm.create_from_mesh(P.tess, P.conserved(), P.gamma, precision=prec)
        if prec == "fp64":
            t = amm.amm_autotune(ctx, 0.3, reps=2)
            assert t["flux_block"] in (64, 128, 256) and amm.amm_get_tuning(ctx)["flux_block"] == t["flux_block"]
            amm.amm_set_tuning(ctx, 4, 4, 64, 0)
        else:
            assert amm.amm_get_tuning(ctx)["flux_block"] == 256
            with pytest.raises(amm.AmmError) as e:
                amm.amm_set_tuning(ctx, 4, 4, 64, 0)
            assert e.value.code == amm.AMM_ERR_INVALID_ARG
