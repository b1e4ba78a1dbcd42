"""A 2D tessellation of more generators than 2^31 half-face places hold cells
(32 each): 8200^2 generators of a jittered lattice.  Every cell closes, the
volumes fill the box, and a generic periodic planar mesh has three faces per
cell."""
import pytest

from tests.test_gpu_voronoi import amm  # noqa: F401

pytestmark = pytest.mark.gpu
M = 8200


def test_more_cells_than_places_in_31_bits(amm):  # noqa: F811
    import torch
    n = M * M
    assert 32 * n > 2 ** 31
    if torch.cuda.mem_get_info()[0] < 160 << 30:
        pytest.skip("needs 160 GB of free device memory")
    g = torch.Generator(device="cuda").manual_seed(3)
    k = torch.arange(n, device="cuda")
    p = torch.stack([k // M, k % M], 1).double()
    p += 0.5 + 0.3 * (2 * torch.rand(n, 2, device="cuda", dtype=torch.float64, generator=g) - 1)
    p /= M
    torch.cuda.synchronize()
    t = amm.amm_tess_build(2, n, p.data_ptr(), [1.0, 1.0])
    assert t.n_faces == 3 * n
    assert t.check()[0] == 0

    class View:
        __cuda_array_interface__ = {"shape": (n,), "typestr": "<f8", "data": (int(t.device_cells()[0]), False),
                                    "version": 2}
    vol = torch.as_tensor(View(), device="cuda")
    assert abs(float(vol.sum()) - 1.0) < 1e-9 and float(vol.min()) > 0   # (pairwise sum of 6.7e7 positive terms)
    del vol
