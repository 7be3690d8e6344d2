"""The pair force with two lanes per particle (small groups) gives the bits of
the one-lane form, which the same body meets in a batch of over 100 000
particles; sizes around a warp's sixteen particles and a block's 128."""
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


def body(n, seed):
    rng = np.random.default_rng(seed)
    b = pkg.Body(*W.cube_mesh(0.5), 0.08, 0.104)
    b.set_particles(rng.uniform(-0.48, 0.48, (n, 3)).astype(np.float32),
                    rng.choice([W.CLS_V, W.CLS_I, W.CLS_S], n, p=[0.8, 0.1, 0.1]).astype(np.int32))
    return b


@pytest.mark.parametrize("morton", [False, True])
@pytest.mark.parametrize("n", [1, 9, 10, 11, 15, 16, 17, 79, 80, 81, 127, 128, 129, 2500])
def test_small_group_has_the_bits_of_a_large_one(n, morton):
    small, large = body(n, n), body(n, n)
    rest = body(100001 - n, 7)                # one past the small form's range
    for group in ([small], [rest, large]):
        bt = pkg.Batch(group)
        bt.set_cell_order(morton)
        bt.relax(3, use_graph=False)
        bt.store()
    assert all(np.array_equal(a, b) for a, b in zip(small.get_particles(), large.get_particles()))
