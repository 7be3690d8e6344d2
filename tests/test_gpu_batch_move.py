"""Batch store and load move every body in launches of many bodies at once."""
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


# launches hold 96 bodies; 0 marks an empty body
@pytest.mark.parametrize("counts", [[1], [0, 5, 0, 300, 1], [7] * 96, [3] * 97, [11, 0] * 100])
def test_store_and_load_move_each_body_its_own_state(counts):
    rng = np.random.default_rng(len(counts))
    v, t = W.cube_mesh(0.5)
    xyz = [rng.uniform(-0.4, 0.4, (n, 3)).astype(np.float32) for n in counts]
    cls = [rng.choice([W.CLS_V, W.CLS_I], n).astype(np.int32) for n in counts]
    bodies, plain = [], []
    for x, c in zip(xyz, cls):
        for group in (bodies, plain):
            b = pkg.Body(v, t, 0.1, 0.13)
            b.set_particles(x, c)
            group.append(b)
    bt = pkg.Batch(bodies)
    for again in range(2):
        bt.relax(2, use_graph=False)
        bt.store()
        for b, p, x, c in zip(bodies, plain, xyz, cls):
            p.relax(2)
            got, want = b.get_particles(), p.get_particles()
            assert all(np.array_equal(g, w) for g, w in zip(got, want))
            # the next round starts from other positions, loaded into the batch
            y = (x * np.float32(0.9 - 0.1 * again)).astype(np.float32)
            b.set_particles(y, c)
            p.set_particles(y, c)
        bt.load()
