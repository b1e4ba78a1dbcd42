"""The first cycle of individual time steps of a context, whose own stream is not
ordered after the legacy one, while that one is busy: bins, counters and state
are those of an idle device.  (Its buffers are set up on the context's stream; the call
reads its status behind the legacy stream in the end.)"""
import numpy as np
import pytest

from harness import ics
from tests.test_gpu_individual import amm  # noqa: F401

pytestmark = pytest.mark.gpu


def test_a_busy_legacy_stream_does_not_reach_the_cycle(amm):  # noqa: F811
    import torch
    P = ics.lognormal_3d(12, seed=4)
    Q = P.conserved()

    def cycle(busy):
        ctx = amm.create_from_mesh(P.tess, Q, P.gamma, precision="fp64", mesh_motion="eulerian")
        done = torch.cuda.Event()
        torch.cuda.synchronize()
        if busy:
            torch.cuda._sleep(1_000_000_000)   # about half a second
            done.record()
            assert not done.query()
        st = amm.amm_advance_individual(ctx, 0.3, 4e-3, 30, True)
        out = amm.amm_get_bins(ctx), amm.amm_get_state(ctx), st
        torch.cuda.synchronize()
        amm.amm_destroy(ctx)
        return out

    cycle(False)
    want = cycle(False)
    got = cycle(True)
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
    assert all(got[2][k] == want[2][k] for k in ("substeps", "face_fluxes", "activations"))
