"""The training kernels at their edges: CTAs that take several 128-sample
tiles (two per SM, so from 39 thousand samples on), a batch of one sample and
of whole tiles, an index list; and the Adam step taken with the reduced
gradient."""
import numpy as np
import pytest

from oracle import mlp as M
from tests.test_gpu_mlp import _blocks, _entrywise, backward_bf16, bf16, env  # noqa: F401

pytestmark = pytest.mark.gpu


def network(seed):
    rng = np.random.default_rng(seed)
    p = M.init_params(rng)
    for k in p:
        p[k] = (p[k] + 0.1 * rng.normal(size=p[k].shape)).astype(np.float32).astype(np.float64)
    return {k: bf16(v) if k in ("W1", "W2", "W3") else v for k, v in p.items()}, rng


@pytest.mark.parametrize("n,index", [(1, False), (128, False), (256, True), (38912, False), (78001, True)])
def test_gradients_over_many_tiles(env, n, index):  # noqa: F811
    """Within 5e-4 of the FP64 evaluation at the kernel's BF16 rounding points,
    relative to the sum of the magnitudes of an entry's terms (FP32
    accumulation and rare one-ulp differences of a rounding, as for a single
    tile)."""
    torch, amm = env
    p, rng = network(n)
    rows = n + 50 if index else n
    x, t = bf16(rng.normal(size=(rows, 6))), rng.normal(size=rows).astype(np.float32).astype(np.float64)
    idx = rng.permutation(rows)[:n].astype(np.int32) if index else np.arange(n, dtype=np.int32)
    net = amm.amm_mlp_create(1.4)
    amm.amm_mlp_set_params(net, amm.pack_params(p))
    xd, td = torch.from_numpy(x.astype(np.float32)).cuda(), torch.from_numpy(t.astype(np.float32)).cuda()
    di = torch.from_numpy(idx).cuda()
    g, loss = amm.amm_mlp_grads(net, xd.data_ptr(), td.data_ptr(), di.data_ptr() if index else 0, n)
    ref, S = backward_bf16(p, x[idx], t[idx])
    got = _blocks(g)
    for k in ref:
        assert _entrywise(got[k], ref[k], S[k]) < 5e-4, k
    y = M.forward(p, x[idx])[0]
    assert abs(loss - np.mean((y - t[idx]) ** 2)) < 2e-2 * loss
    # the same batch again: bit for bit
    g2, loss2 = amm.amm_mlp_grads(net, xd.data_ptr(), td.data_ptr(), di.data_ptr() if index else 0, n)
    assert np.array_equal(g, g2) and loss == loss2


def test_adam_step_follows_the_gradient(env):  # noqa: F811
    """Three steps: the parameters move by Adam with the gradients that
    amm_mlp_grads reports, to FP32 rounding (a step is at most a few lr, the
    parameters of order one), and the next gradient is taken at the new
    weights."""
    torch, amm = env
    p, rng = network(5)
    n, lr = 700, 1e-3
    x, t = rng.normal(size=(n, 6)).astype(np.float32), rng.normal(size=n).astype(np.float32)
    xd, td = torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda()
    net = amm.amm_mlp_create(1.4)
    amm.amm_mlp_set_params(net, amm.pack_params(p))
    m = v = np.zeros(amm.amm_mlp_num_params())
    for k in range(1, 4):
        before = amm.amm_mlp_get_params(net).astype(np.float64)
        g, loss = amm.amm_mlp_grads(net, xd.data_ptr(), td.data_ptr(), 0, n)
        lossd = torch.zeros(1, device="cuda")
        amm.amm_mlp_train_step(net, xd.data_ptr(), td.data_ptr(), 0, n, lr, lossd.data_ptr())
        amm.amm_mlp_sync(net)
        g = g.astype(np.float64)
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        step = lr * (m / (1 - 0.9 ** k)) / (np.sqrt(v / (1 - 0.999 ** k)) + 1e-8)
        after = amm.amm_mlp_get_params(net).astype(np.float64)
        assert np.max(np.abs(after - (before - step))) < 2.0 ** -23 * np.abs(before).max() + 1e-4 * lr
        assert float(lossd.item()) == loss
