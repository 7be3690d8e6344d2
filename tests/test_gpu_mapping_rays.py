"""The crossing test of the generation rays ends most triangles in FP32 where
two edges are certainly on opposite sides; the classes stay those of the FP64
test, also where rays meet vertices and edges to within FP32 rounding, close
to the origin and far from it (the ray's offset is then below an ulp)."""
import numpy as np
import pytest

import oracle as O
import paper_2501_03056_gb300 as pkg
from paper_2501_03056_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2501_03056_gb300 import _build
    _build.build()


def slab(n, x, y, rng):
    """A slab with n x n vertices (x, y) on either side, closed around."""
    k = np.arange(n * n).reshape(n, n)
    a, b, c, d = k[:-1, :-1].ravel(), k[1:, :-1].ravel(), k[1:, 1:].ravel(), k[:-1, 1:].ravel()
    top = np.concatenate([np.stack([a, b, c], 1), np.stack([a, c, d], 1)])
    rim = np.concatenate([k[:-1, 0], k[-1, :-1], k[:0:-1, -1], k[0, :0:-1]])
    nxt, low = np.roll(rim, -1), n * n
    side = np.concatenate([np.stack([rim, rim + low, nxt + low], 1), np.stack([rim, nxt + low, nxt], 1)])
    z = np.concatenate([0.3 + 0.08 * rng.random(n * n), -0.3 - 0.08 * rng.random(n * n)])
    v = np.stack([np.tile(x.ravel(), 2), np.tile(y.ravel(), 2), z], 1).astype(np.float32)
    return v, np.concatenate([top, (top + low)[:, ::-1], side]).astype(np.int32)


@pytest.mark.parametrize("shift", [0.0, 3.7, 250.0])
@pytest.mark.parametrize("on_rays", [0.0, 0.5, 1.0])
def test_rays_through_vertices_and_edges(shift, on_rays):
    rng = np.random.default_rng(3)
    n, dx = 12, 0.05
    x, y = np.meshgrid(np.linspace(0, 1.1, n) + shift, np.linspace(0, 1.1, n) - shift, indexing="ij")
    o = O.Oracle(*slab(n, x, y, rng), dx, 1.3 * dx).tri_grid()[0]
    # the inner vertices on the rays nearest to them
    inner = np.zeros((n, n), bool)
    inner[1:-1, 1:-1] = rng.random((n - 2, n - 2)) < on_rays
    for p, k, off in ((x, 0, 1.234567e-6), (y, 1, 2.345678e-6)):
        cell = np.floor((p - o[k]) / dx)
        ray = (o[k] + (cell + 0.5) * dx).astype(np.float32).astype(np.float64) + off * dx
        p[inner] = ray[inner]
    v, t = slab(n, x, y, rng)
    b, orc = pkg.Body(v, t, dx, 1.3 * dx), O.Oracle(v, t, dx, 1.3 * dx)
    assert np.array_equal(orc.tri_grid()[0][:2], o[:2])
    m = b.map_particles(surface=False)
    px, pc, _ = b.get_particles()
    ox, oc, _ = orc.map_particles(surface=False)
    assert m == len(ox) > 1000 and np.array_equal(pc, oc)
    assert np.abs(px.astype(np.float64) - ox).max() < 1e-6 * max(1.0, np.abs(ox).max())
