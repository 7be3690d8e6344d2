"""Generation on word bitmaps against the oracle: rows that end inside, at and
just past a word, columns that a slanted or folded surface crosses many times,
bands from one cell to more than a word, and a second generation of the same
body."""
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


def turned(v, angle):
    c, s = np.cos(angle), np.sin(angle)
    r = np.array([[c, -s, 0], [s, c, 0], [0, 0, 1]]) @ np.array([[1, 0, 0], [0, c, -s], [0, s, c]])
    return (v.astype(np.float64) @ r.T).astype(np.float32)


def check(b, o, **options):
    n = b.map_particles(**options)
    x, c, cons = b.get_particles()
    ox, oc, ocons = o.map_particles(**options)
    assert n == len(ox) and np.array_equal(c, oc)
    s = c == W.CLS_S
    assert s.sum() == 0 or (cons[s] == ocons[s]).mean() > 0.995
    assert len(ox) == 0 or np.abs(x.astype(np.float64) - ox).max() < 1e-6 * max(1.0, np.abs(ox).max())


# the triangle grid has 4 to 5 cells of margin along x: rows of 30 to 34 and
# of 62 to 66 cells, and a body narrower than a word
@pytest.mark.parametrize("cells_x", [3, 26, 27, 28, 29, 58, 59, 60, 61])
def test_rows_around_a_word(cells_x):
    v, t = W.cube_mesh(0.5)
    dx = 0.05
    v = (v * np.array([cells_x * dx * 1.003, 0.41, 0.53])).astype(np.float32)
    b, o = pkg.Body(v, t, dx, 1.3 * dx), O.Oracle(v, t, dx, 1.3 * dx)
    check(b, o)
    check(b, o, band_cells=1, inner_cells=1)
    check(b, o, surface=False, features=False)
    check(b, o, volume=False)


@pytest.mark.parametrize("mesh,options", [
    ("gear", {"band_cells": 2, "inner_cells": 1}), ("torus", {}), ("torus", {"band_cells": 3, "inner_cells": 2}),
    ("cylinder", {"band_cells": 1})])
def test_turned_bodies_and_bands(mesh, options):
    if mesh == "gear":
        v, t = W.gear_mesh(teeth=12, r_out=0.5, r_root=0.42, r_bore=0.15, height=0.2, pts_per_tooth=3, rings=4, nz=3,
                           bore_points=36)
        dx = 0.026
    elif mesh == "torus":
        v, t = W.torus_mesh(1.0, 0.3, 64, 24)
        dx = 0.06
    else:
        v, t = W.cylinder_mesh(0.5, 1.0, 48, 4)
        dx = 0.05
    v = turned(v, 0.73)
    b, o = pkg.Body(v, t, dx, 1.3 * dx), O.Oracle(v, t, dx, 1.3 * dx)
    assert b.extract_features(30.0) == o.extract_features(30.0)
    for _ in range(2):                 # the second generation reuses the arrays
        check(b, o, **options)


def test_bands_wider_than_a_word():
    # a cube of 77 cells: the band is a shell of its cells along each axis
    v, t = W.cube_mesh(0.5)
    dx = 0.05
    b = pkg.Body((v * np.float32(77 * dx * 1.003)).astype(np.float32), t, dx, 1.3 * dx)
    b.map_particles(surface=False)
    x0, c0, _ = b.get_particles()
    depth = 0.5 * 77 * dx * 1.003 - np.abs(x0).max(axis=1)
    for band in (31, 32, 33):
        b.map_particles(surface=False, band_cells=band)
        x, c, _ = b.get_particles()
        assert np.array_equal(x, x0)
        # depth in cells of a cell centre below the nearest face, to half a cell
        k = depth / dx
        assert (c[k < band - 0.6] == W.CLS_V).all() and (c[k > band + 1.6] == W.CLS_I).all()
        assert (c == W.CLS_V).any() and (c == W.CLS_I).any()
    b.map_particles(surface=False, band_cells=64, inner_cells=64)
    assert (b.get_particles()[1] == W.CLS_V).all()
