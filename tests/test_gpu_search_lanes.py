"""The triangle search with 1, 8 or 32 lanes per particle gives the same bits,
on meshes whose candidate lists are short, long and too long to merge (their
27 cells are probed), with both projection rules, with Boolean partners and
with feature lines long enough to be searched too."""
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


def bodies(kind, cascade):
    if kind == "cube":                       # lists of one or two triangles: 8 lanes
        mesh, dx = W.cube_mesh(0.5), 0.06
    elif kind == "rims":                     # feature lines of 9 and 96 segments, in the search
        mesh, dx = W.cylinder_mesh(0.5, 1.0, 96 if not cascade else 9, 4), 0.06
    elif kind == "sphere":                   # lists of about a hundred: 32 lanes
        mesh, dx = W.icosphere_mesh(4, 0.5), 0.08
    else:                                    # "probe": over 512 entries in the 27 cells
        mesh, dx = W.icosphere_mesh(5, 0.5), 0.15
    b = pkg.Body(*mesh, dx, 1.3 * dx)
    b.extract_features(30.0)
    b.map_particles()
    out = [b]
    if kind == "cube":                       # united with a sphere through its side
        v, t = W.icosphere_mesh(2, 0.3)
        c = pkg.Body((v + np.array([0.45, 0.03, -0.02])).astype(np.float32), t, dx, 1.3 * dx)
        c.map_particles()
        pkg.union(b, c)
        out.append(c)
    rng = np.random.default_rng(4)
    for q in out:
        q.set_projection_rule(cascade)
        x, cls, cons = q.get_particles()
        x = x + (rng.uniform(-0.2, 0.2, x.shape) * dx * (cls == W.CLS_V)[:, None]).astype(np.float32)
        q.set_particles(x, cls)
        q.set_constraints(cons)
    return out


@pytest.mark.parametrize("cascade", [False, True])
@pytest.mark.parametrize("kind", ["cube", "rims", "sphere", "probe"])
def test_lanes_do_not_change_the_search(kind, cascade):
    got = []
    for ctas in (0, 1, 8):
        bs = bodies(kind, cascade)
        if kind == "probe":
            assert bs[0].debug_cell_lists()[2] > 0
        bt = pkg.Batch(bs)
        bt.configure(0, 256, ctas)
        bt.relax(4, use_graph=False)
        bt.store()
        got.append([a for b in bs for a in b.get_particles()])
    for other in got[1:]:
        assert all(np.array_equal(a, b) for a, b in zip(got[0], other))


# every mesh with every number of lanes, whatever the library would take
@pytest.mark.parametrize("cascade", [False, True])
@pytest.mark.parametrize("kind", ["cube", "rims", "sphere", "probe"])
def test_each_number_of_lanes_gives_the_same_bits(kind, cascade):
    got = []
    for lanes in (1, 8, 32):
        bs = bodies(kind, cascade)
        bt = pkg.Batch(bs)
        assert bt.debug_search_lanes(lanes) == lanes
        bt.relax(4, use_graph=False)
        bt.store()
        got.append([a for b in bs for a in b.get_particles()])
    for other in got[1:]:
        assert all(np.array_equal(a, b) for a, b in zip(got[0], other))


def cloud_in(mesh, dx, n=2000):
    b = pkg.Body(*mesh, dx, 1.3 * dx)
    b.set_particles(np.random.default_rng(n).uniform(-0.2, 0.2, (n, 3)).astype(np.float32), np.full(n, W.CLS_V, np.int32))
    return b


def test_cells_too_long_for_a_list_count_with_their_length():
    short = cloud_in(W.cube_mesh(0.5), 0.06)
    assert pkg.Batch([short]).debug_search_lanes() == 8
    # 5,120 triangles within a few cells: no cell has a list, every one is probed
    dense = cloud_in(W.icosphere_mesh(4, 0.05), 0.2)
    cells, entries, probed = dense.debug_cell_lists()
    assert probed > 0 and entries < 8 * cells
    assert pkg.Batch([dense]).debug_search_lanes() == 32
    # one such mesh among bodies of short lists: its particles walk longest
    flat = [cloud_in(W.cube_mesh(2.0), 0.02, 3000) for _ in range(2)]
    mixed = flat + [dense]
    c, e = (sum(b.debug_cell_lists()[k] for b in mixed) for k in (0, 1))
    assert e + 27 * 5120 * probed < 8 * c
    assert pkg.Batch(flat).debug_search_lanes() == 8
    assert pkg.Batch(mixed).debug_search_lanes() == 32


def test_lanes_are_checked():
    bt = pkg.Batch([cloud_in(W.cube_mesh(0.5), 0.06)])
    for bad in (-1, 2, 16, 64):
        with pytest.raises(pkg.FPPGError) as e:
            bt.debug_search_lanes(bad)
        assert e.value.code == pkg.ERR_ARG
