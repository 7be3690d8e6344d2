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


def test_fixed_particles_on_one_key_take_linear_time():
    # twice as many on the key: far from four times as long (ranking each
    # against all takes 3.8 times as long from 100,000 to 200,000)
    import torch
    v, t = W.cube_mesh(0.5)
    took = []
    for n in (100000, 200000):
        b = pkg.Body(v, t, 0.02, 0.026, stream=torch.cuda.current_stream())
        b.set_particles(np.full((n, 3), 0.1234, np.float32), np.full(n, W.CLS_I, np.int32))
        b.relax(1)
        runs = []
        for _ in range(5):
            t0, t1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            t0.record()
            b.relax(2)
            t1.record()
            t1.synchronize()
            runs.append(t0.elapsed_time(t1))
        took.append(sorted(runs)[2])
    assert took[1] < 2.9 * took[0]


def test_few_particles_on_a_large_grid_are_not_slower_than_by_the_radix_sort():
    # 3.9 M fine keys, whose counts were cleared by the blocks of the particles:
    # 273 us an iteration, the radix sort 79
    import torch
    v, t = W.cube_mesh(0.5)
    rng = np.random.default_rng(2)
    took = []
    for counted in (None, False):
        b = pkg.Body(v, t, 0.005, 0.0065, stream=torch.cuda.current_stream())
        b.set_particles(rng.uniform(-0.5, 0.5, (100, 3)).astype(np.float32), np.full(100, W.CLS_V, np.int32))
        if counted is not None:
            b.set_incremental(counted)
        b.relax(2)
        runs = []
        for _ in range(5):
            t0, t1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            t0.record()
            b.relax(20)
            t1.record()
            t1.synchronize()
            runs.append(t0.elapsed_time(t1))
        took.append(sorted(runs)[2])
    assert took[0] < 1.2 * took[1]


# a set that crowds a key when it is given takes the radix sort, and only that
# one: at the edge (512), for a batch when it is made and when it is loaded again
@pytest.mark.parametrize("m,crowded", [(512, False), (513, True), (20000, True)])
def test_a_crowded_set_is_ordered_by_the_radix_sort(m, crowded):
    rng = np.random.default_rng(m)
    v, t = W.cube_mesh(0.5)
    loose = rng.uniform(-0.45, 0.45, (25000, 3)).astype(np.float32)
    tight = loose.copy()
    tight[rng.permutation(len(loose))[:m]] = 0.49        # (a key that holds no other)
    cls = np.where(rng.uniform(size=len(loose)) < 0.5, W.CLS_I, W.CLS_P).astype(np.int32)

    def body(x):
        b = pkg.Body(v, t, 0.05, 0.065)
        b.set_particles(x, cls)
        return b

    kernels = pkg.Batch([body(loose)]).kernels_per_iter
    radix = pkg.Batch([body(loose)])
    radix.set_incremental(False)
    assert radix.kernels_per_iter > kernels
    a, b = body(loose), body(tight)
    bt = pkg.Batch([a, b])
    assert (bt.kernels_per_iter == kernels) == (not crowded)
    b.set_particles(loose, cls)
    bt.load()
    assert bt.kernels_per_iter == kernels
    b.set_particles(tight, cls)
    bt.load()
    assert (bt.kernels_per_iter == kernels) == (not crowded)
    bt.set_graph_iters(2)
    bt.relax(2, use_graph=True)
    bt.autotune(1)
    assert (bt.kernels_per_iter == kernels) == (not crowded)
    # moving classes on one key that stop moving, in a body and in a batch
    b = pkg.Body(v, t, 0.05, 0.065)
    b.set_particles(tight, np.full(len(tight), W.CLS_V, np.int32))
    moving = pkg.Batch([b])
    assert moving.kernels_per_iter == kernels
    moving.set_mobile_classes((W.CLS_S, W.CLS_F))
    assert (moving.kernels_per_iter == kernels) == (not crowded)
    b.set_mobile_classes((W.CLS_S, W.CLS_F))
    assert (pkg.Batch([b]).kernels_per_iter == kernels) == (not crowded)
    b = pkg.Body(v, t, 0.05, 0.065)
    b.set_particles(tight, np.full(len(tight), W.CLS_V, np.int32))
    b.set_ghost_count(len(tight))
    assert (pkg.Batch([b]).kernels_per_iter == kernels) == (not crowded)
    b, bt = body(tight), pkg.Batch([a, body(loose)])
    bt.set_incremental(True)                      # the caller's choice stands
    bt.load()
    assert bt.kernels_per_iter == kernels
    loaded = pkg.Batch([b])
    loaded.set_incremental(True)
    loaded.load()
    assert loaded.kernels_per_iter == kernels


@pytest.mark.parametrize("kind,m,fixed,crowded", [
    ("joined", 400, False, False), ("joined", 600, False, True), ("loose", 600, False, False),
    ("loose", 600, True, True), ("loose", 400, True, False)])
def test_features_on_one_key_are_noticed_when_they_are_generated(kind, m, fixed, crowded):
    # tiny triangles within a thousandth of dx: m pairs joined at a corner, which
    # is a singular point (fixed), or m loose ones, each a loop with one feature
    # point (fixed on request)
    dx = 0.1
    rng = np.random.default_rng(8)
    c = rng.uniform(-1e-4, 1e-4, (m, 3)) + 0.03
    v = np.concatenate([c] + [c + rng.normal(size=(m, 3)) * 1e-5 for _ in range(4)])
    k = np.arange(m)
    t = [np.stack([k, k + m, k + 2 * m], 1)] + [np.stack([k, k + 3 * m, k + 4 * m], 1)] * (kind == "joined")
    t = np.concatenate(t + [[[5 * m, 5 * m + 1, 5 * m + 2]]])
    v = np.concatenate([v, [[-1.0, -1, -1], [1, 1, 1], [1, -1, 1]]])
    b = pkg.Body(v.astype(np.float32), t.astype(np.int32), dx, 1.3 * dx)
    b.set_fixed_features(fixed)
    b.extract_features(30.0)
    b.map_particles(surface=False, volume=False)
    n = np.bincount(b.get_particles()[1], minlength=5)
    assert n[W.CLS_P] == (m if kind == "joined" else 0) and n[W.CLS_F] >= (0 if kind == "joined" else m)
    radix = pkg.Batch([b])
    radix.set_incremental(False)
    assert (pkg.Batch([b]).kernels_per_iter == radix.kernels_per_iter) == crowded


def test_looking_for_crowds_waits_for_a_relaxation_on_another_stream():
    # 20,000 fixed particles among moving ones; the classes are set again on
    # another stream while the body relaxes
    import torch
    rng = np.random.default_rng(12)
    x = rng.uniform(-0.45, 0.45, (40000, 3)).astype(np.float32)
    cls = np.where(rng.uniform(size=len(x)) < 0.5, W.CLS_I, W.CLS_V).astype(np.int32)
    got = []
    for switch in (False, True):
        b = pkg.Body(*W.cube_mesh(0.5), 0.03, 0.039)
        b.set_particles(x, cls)
        one, two = torch.cuda.Stream(), torch.cuda.Stream()
        b.set_stream(one)
        b.relax(300)
        if switch:
            b.set_stream(two)
            b.set_mobile_classes((W.CLS_S, W.CLS_V, W.CLS_F))
            b.set_fixed_features(False)
        got.append(b.get_particles()[0])
        b.relax(20)
        got.append(b.get_particles()[0])
    assert np.array_equal(got[0], got[2]) and np.array_equal(got[1], got[3])
