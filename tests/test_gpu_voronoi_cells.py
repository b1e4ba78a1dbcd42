"""The 3D Voronoi cell kernels where they hand over and refuse: cells with
more vertices or planes than the kernel for ordinary cells holds (a generator
inside a sphere of 44 others; two skew rows of generators, every pair of which
shares a face, whose half-faces also outgrow the list's first allocation),
random generators (shells beyond the first), boxes of a few generators (cells
that meet their own images), an exact lattice (four planes through a point),
and uneven box lengths -- each against the host tessellator: the same faces,
areas and centroids to 1e-9 of the mean face scale, the neighbours of every
cell counted alike."""
import numpy as np
import pytest

from harness import ics
from harness.tess import tessellate
from tests.test_gpu_voronoi import amm, face_key_map, gpu_tess  # noqa: F401

pytestmark = pytest.mark.gpu


def sphere(m=44):
    rng = np.random.default_rng(5)
    k = np.arange(m) + 0.5
    ph, th = np.arccos(1 - 2 * k / m), np.pi * (1 + 5 ** 0.5) * k
    s = 0.5 + 0.2 * np.column_stack([np.cos(th) * np.sin(ph), np.sin(th) * np.sin(ph), np.cos(ph)])
    s += rng.uniform(-1e-3, 1e-3, (m, 3))
    o = rng.uniform(0, 1, (300, 3))
    return np.concatenate([[[0.5, 0.5, 0.5]], s, o[np.linalg.norm(o - 0.5, axis=1) > 0.33]]), np.ones(3)


def skew(c=4, m=13):
    rng = np.random.default_rng(6)
    t = (np.arange(m) + 0.5) / m - 0.5
    one = 0.5 + np.concatenate([np.column_stack([0.8 * t, 0 * t, 0 * t + 0.12]),
                                np.column_stack([0 * t, 0.8 * t, 0 * t - 0.12])])
    g = np.stack(np.meshgrid(*[np.arange(c)] * 3, indexing="ij"), -1).reshape(-1, 1, 3)
    p = (g + one[None]).reshape(-1, 3) + rng.uniform(-1e-4, 1e-4, (c ** 3 * 2 * m, 3))
    return p / c, np.ones(3)


def lattice(n, jitter, box=(1.0, 1.0, 1.0), seed=1):
    return ics.jittered_lattice((n,) * 3, np.array(box), jitter, np.random.default_rng(seed)), np.array(box)


MESHES = {
    "sphere": sphere, "skew": skew, "random": lambda: (np.random.default_rng(2).uniform(0, 1, (2500, 3)), np.ones(3)),
    "few": lambda: lattice(2, 0.3), "exact": lambda: lattice(6, 0.0), "almost": lambda: lattice(7, 1e-9), "uneven": lambda: lattice(8, 0.4, (1.0, 0.3, 2.0)),
    "small": lambda: lattice(6, 0.3, (1e-9, 2e-9, 1e-9)),
}


@pytest.mark.parametrize("name", sorted(MESHES))
def test_cells_match_the_host(amm, name):  # noqa: F811
    pts, box = MESHES[name]()
    H = tessellate(pts, box)
    t, (cells, shift, area, cen, vol, com) = gpu_tess(amm, pts, box)
    mh, mg = face_key_map(H.cells, H.shift, H.area, H.centroid), face_key_map(cells, shift, area, cen)
    scale = np.mean(H.area)
    # (a face of almost no area may be listed by one and not the other)
    odd = [max(mh.get(k, (0,))[0], mg.get(k, (0,))[0]) for k in set(mh) ^ set(mg)]
    assert max(odd, default=0.0) < 1e-9 * scale
    for k in set(mh) & set(mg):
        assert abs(mg[k][0] - mh[k][0]) < 1e-9 * scale
        assert np.abs(mg[k][1] - mh[k][1]).max() < 1e-9 * np.sqrt(scale) or mh[k][0] < 1e-6 * scale
    np.testing.assert_allclose(vol, H.volume, rtol=1e-9)
    assert t.check()[0] <= len(odd)
    if name in ("sphere", "skew"):
        assert H.faces_per_cell.max() > 34   # more than 64 vertices (2 F - 4)


def test_refusals_stay(amm):  # noqa: F811
    """A generator outside the box; a box too sparse for its cells to close."""
    pts, box = lattice(5, 0.2)
    far = pts.copy()
    far[7, 1] = 1.0
    lone = np.random.default_rng(3).uniform(0, 1, (9, 3))
    for p, code in ((far, amm.AMM_ERR_INVALID_ARG), (lone, amm.AMM_ERR_NUMERIC)):
        with pytest.raises(amm.AmmError) as e:
            gpu_tess(amm, p, box)
        assert e.value.code == code
    gpu_tess(amm, pts, box)
