"""The counting sort over the fine keys against the radix sort.

Both give the one order by (key, id) and the start table of the fine keys:
keys, permutation, cell ranges and a relaxed state are the same bits, at the
edges of the tiles (of particles and of keys), on keys shared by many
particles, on clouds clamped into the boundary cells, in both row orders and
on grids large enough for every way of adding up the counts."""
import numpy as np
import pytest

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


def cloud(kind, n, rng):
    if kind == "uniform":
        return rng.uniform(-0.5, 0.5, (n, 3))
    if kind == "shared":              # hundreds to thousands of particles per key, shuffled ids
        x = np.concatenate([np.full((n // 2, 3), 0.1234), rng.uniform(0.2, 0.22, (n - n // 2, 3))])
        return x[rng.permutation(n)]
    return rng.uniform(-3.0, 3.0, (n, 3))      # "outside": mostly clamped


def both_orders(xyz, cls, dx, order, grid):
    v, t = W.cube_mesh(0.5)
    out = []
    for counted in (True, False):
        b = pkg.Body(v, t, dx, 1.3 * dx)
        b.set_particles(xyz, cls)
        b.set_incremental(counted)
        b.set_cell_order(order)
        got = list(b.debug_grid()) if grid else []
        b.relax(2)
        got.append(b.get_particles()[0])
        b.relax(1)
        got.append(b.get_particles()[0])
        out.append(got)
    return out


@pytest.mark.parametrize("order", [pkg.ORDER_ROWS, pkg.ORDER_MORTON_ROWS])
@pytest.mark.parametrize("kind,n,dx", [
    ("uniform", 1, 0.05), ("uniform", 2, 0.05), ("uniform", 255, 0.05), ("uniform", 512, 0.05),
    ("uniform", 513, 0.02), ("uniform", 20001, 0.02), ("shared", 5001, 0.05), ("outside", 7000, 0.04)])
def test_counting_sort_equals_the_radix_sort(kind, n, dx, order):
    rng = np.random.default_rng(n)
    xyz = cloud(kind, n, rng).astype(np.float32)
    a, b = both_orders(xyz, rng.integers(0, 5, n).astype(np.int32), dx, order, True)
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


def test_counting_sort_with_two_particles_per_thread():
    rng = np.random.default_rng(9)
    xyz = rng.uniform(-0.5, 0.5, ((1 << 20) + 257, 3)).astype(np.float32)
    a, b = both_orders(xyz, rng.integers(0, 5, len(xyz)).astype(np.int32), 0.01, pkg.ORDER_ROWS, True)
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


def test_counting_sort_on_a_grid_of_more_tiles_than_a_block_adds_up():
    # 8.5 M cells: 68 M fine keys in 16,600 tiles, whose sums are scanned
    rng = np.random.default_rng(5)
    xyz = rng.uniform(-0.5, 0.5, (30001, 3)).astype(np.float32)
    a, b = both_orders(xyz, np.full(len(xyz), W.CLS_V, np.int32), 0.00188, pkg.ORDER_ROWS, True)
    assert len(a[2]) > 25000
    for x, y in zip(a, b):
        assert np.array_equal(x, y)
