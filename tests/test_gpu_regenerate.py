"""Generating again at the same particle count uses the body's arrays again: the
new set is that of a fresh body, whatever the old one went through, also when
the body was still relaxing on another stream."""
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


def body():
    v, t = W.cylinder_mesh(0.5, 1.0, 64, 4)
    b = pkg.Body(v, t, 0.02, float(np.float32(1.3 * 0.02)))
    b.extract_features(30.0)
    b.map_particles(band_cells=3)
    return b


@pytest.mark.parametrize("iters,switch", [(20, False), (400, True)])
def test_the_second_generation_is_the_first(iters, switch):
    import torch
    fresh = body()
    x0, cls, cons = fresh.get_particles()
    fresh.relax(3)                      # certificates and maxima of a first relaxation
    want = [x0, cls, cons, *fresh.get_particles()]
    b = body()
    if switch:
        one, two = torch.cuda.Stream(), torch.cuda.Stream()
        b.set_stream(one)
        b.relax(iters)                  # still under way when the set is made anew
        b.set_stream(two)
    else:
        b.relax(iters)
    assert b.map_particles(band_cells=3) == len(x0)
    got = list(b.get_particles())
    b.relax(3)
    got += b.get_particles()
    assert all(np.array_equal(g, w) for g, w in zip(got, want))
    assert b.stats() == fresh.stats()
