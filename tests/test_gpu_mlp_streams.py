"""A network made on a stream that is not ordered after the legacy one, while
that one is busy: weights set, evaluated and trained give what they give on an
idle device.  (All buffers are cleared when amm_mlp_create and the first
training call return, so nothing lands later.)"""
import numpy as np
import pytest

from oracle import mlp as M
from tests.test_gpu_mlp import env  # noqa: F401
from tests.test_gpu_mlp_tiles import network

pytestmark = pytest.mark.gpu


def test_a_busy_legacy_stream_does_not_reach_the_network(env):  # noqa: F811
    torch, amm = env
    p, rng = network(5)
    packed = amm.pack_params(p)
    x = torch.from_numpy(rng.normal(size=(256, 6)).astype(np.float32)).cuda()
    t = torch.from_numpy(rng.normal(size=256).astype(np.float32)).cuda()
    torch.cuda.synchronize()

    def use(stream):
        net = amm.amm_mlp_create(1.4, stream)
        amm.amm_mlp_set_params(net, packed)
        y = torch.empty(256, device="cuda")
        amm.amm_mlp_forward(net, x.data_ptr(), 256, y.data_ptr())
        amm.amm_mlp_train_step(net, x.data_ptr(), t.data_ptr(), 0, 256, 1e-3)
        amm.amm_mlp_sync(net)
        return net, y

    ref_net, ref_y = use(None)
    torch.cuda.synchronize()
    want_y, want_p = ref_y.cpu().numpy(), amm.amm_mlp_get_params(ref_net)
    assert np.abs(want_y - M.forward(p, x.cpu().numpy().astype(np.float64))[0]).max() < 0.1
    side = torch.cuda.Stream()
    assert torch.cuda.current_stream().cuda_stream == 0
    done = torch.cuda.Event()
    torch.cuda._sleep(400_000_000)         # about 0.2 s on the legacy stream
    done.record()
    net, y = use(side.cuda_stream)
    overlapped = not done.query()
    torch.cuda.synchronize()
    assert np.array_equal(y.cpu().numpy(), want_y)
    assert np.array_equal(amm.amm_mlp_get_params(net), want_p)
    # and nothing arrived afterwards
    amm.amm_mlp_forward(net, x.data_ptr(), 256, y.data_ptr())
    assert np.abs(y.cpu().numpy()).max() > 0
    amm.amm_mlp_set_params(net, packed)
    amm.amm_mlp_forward(net, x.data_ptr(), 256, y.data_ptr())
    assert np.array_equal(y.cpu().numpy(), want_y)
    assert overlapped, "the legacy stream was not busy meanwhile"
