"""The generation counts a ray's crossing of a triangle at the lowest cell of the
column that lists the triangle, and looks for the triangle only in the cell
below.  So the cells of a column that list a triangle have to be one run along z
wherever the column's ray meets the triangle.  The binning's own arithmetic is
checked here (the oracle's FP64 separating-axis test, operation for operation
the library's) on triangles where it could fail: slivers, steep and flat ones,
edges along the axes and on cell faces, corners one rounding apart, far from the
origin and hundreds of cells long."""
import numpy as np
import pytest

import oracle as O


def soup(kind, rng, m, dx):
    """m triangles as (verts [3m, 3], tris [m, 3])"""
    n = {"long": 60, "thin": 60}.get(kind, 12)
    a = rng.uniform(0, n * dx, (m, 3))
    e1, e2 = rng.normal(size=(2, m, 3))
    if kind == "long":
        e1, e2 = e1 * 40 * dx, e2 * 3 * dx
    elif kind == "thin":          # a sliver: its third corner near its longest edge
        e1 = e1 * 30 * dx
        e2 = e1 * rng.uniform(0, 1, (m, 1)) + e2 * dx * 10.0 ** rng.uniform(-7, -1, (m, 1))
    elif kind == "steep":         # almost along z
        e1, e2 = e1 * dx * [0.7, 0.7, 9], e2 * dx * [1e-4, 0.7, 9]
    elif kind == "flat":          # almost across z, through many columns
        e1, e2 = e1 * dx * [6, 6, 1e-7], e2 * dx * [6, 6, 1e-6]
    elif kind == "axes":          # corners on faces and edges of cells, edges along the axes
        a = rng.integers(0, 2 * n, (m, 3)) * (0.5 * dx)
        e1 = rng.integers(-8, 9, (m, 3)) * (0.5 * dx) * (rng.uniform(size=(m, 3)) < 0.6)
        e2 = rng.integers(-8, 9, (m, 3)) * (0.5 * dx) * (rng.uniform(size=(m, 3)) < 0.6)
    else:                         # "rounded": the same, each coordinate a rounding or two off
        v, t = soup("axes", rng, m, dx)
        up = rng.integers(-2, 3, v.shape)
        for _ in range(2):
            v = np.where(up > 0, np.nextafter(v, np.float32(9)), np.where(up < 0, np.nextafter(v, np.float32(-9)), v))
            up = up - np.sign(up)
        return v, t
    v = np.stack([a, a + e1, a + e2], 1).reshape(-1, 3)
    return v.astype(np.float32), np.arange(3 * m, dtype=np.int32).reshape(m, 3)


@pytest.mark.parametrize("kind", ["long", "thin", "steep", "flat", "axes", "rounded"])
@pytest.mark.parametrize("dx,shift", [(0.1, 0.0), (0.0371, 100.0)])
def test_a_triangle_lists_one_run_of_cells_where_the_ray_meets_it(kind, dx, shift):
    rng = np.random.default_rng(len(kind) * 7 + int(100 * dx))
    m = 150 if kind in ("long", "thin") else 400
    v, t = soup(kind, rng, m, dx)
    v = (v + np.float32(shift)).astype(np.float32)
    o = O.Oracle(v, t, dx, 1.3 * dx)
    org, _, n = o.tri_grid()
    ox, oy = float(org[0]), float(org[1])
    key, tri = o.tri_bins()
    nx, ny = int(n[0]), int(n[1])
    x, y, z = key % nx, key // nx % ny, key // (nx * ny)
    d = float(np.float32(dx))
    qx = (ox + (x + 0.5) * d).astype(np.float32).astype(np.float64) + 1.234567e-6 * d
    qy = (oy + (y + 0.5) * d).astype(np.float32).astype(np.float64) + 2.345678e-6 * d
    a, b, c = (v[t[tri, k]].astype(np.float64) for k in range(3))
    area = (b[:, 0] - a[:, 0]) * (c[:, 1] - a[:, 1]) - (c[:, 0] - a[:, 0]) * (b[:, 1] - a[:, 1])
    with np.errstate(all="ignore"):
        l1 = ((b[:, 0] - qx) * (c[:, 1] - qy) - (c[:, 0] - qx) * (b[:, 1] - qy)) / area
        l2 = ((c[:, 0] - qx) * (a[:, 1] - qy) - (a[:, 0] - qx) * (c[:, 1] - qy)) / area
        met = (area != 0) & ~(l1 < 0) & ~(l2 < 0) & ~(1 - l1 - l2 < 0)
    assert met.sum() > 20
    order = np.lexsort((z, y, x, tri))
    order = order[met[order]]
    same = (tri[order][1:] == tri[order][:-1]) & (x[order][1:] == x[order][:-1]) & (y[order][1:] == y[order][:-1])
    assert (np.diff(z[order])[same] == 1).all()
