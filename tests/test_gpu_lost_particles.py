"""A body whose particles are gone, or replaced, after it was batched or between
the two halves of an iteration: every call that would use the old arrays is
refused on the host."""
import ctypes

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
    yield
    pkg.lib().fppg_debug_fail_allocation(-1)


def body(n=500, seed=3):
    v, t = W.cube_mesh(0.5)
    b = pkg.Body(v, t, 0.1, 0.13)
    x = np.random.default_rng(seed).uniform(-0.4, 0.4, (n, 3)).astype(np.float32)
    b.set_particles(x, np.full(n, W.CLS_V, np.int32))
    return b


def held(b):
    n = ctypes.c_int64()
    assert pkg.lib().fppg_get_particles(b.handle, None, None, None, 0, ctypes.byref(n)) == pkg.OK
    return n.value


def lose_by_setting(b):
    b.set_particles(np.zeros((900, 3), np.float32), np.full(900, W.CLS_V, np.int32))


def lose_by_generating(b):
    b.map_particles()


@pytest.mark.parametrize("lose", [lose_by_setting, lose_by_generating])
def test_a_batch_does_not_touch_the_arrays_a_body_lost(lose):
    for k in range(40):                     # every allocation of the call, one after another
        a, b = body(), body(seed=5)
        bt = pkg.Batch([a, b])
        bt.relax(1, use_graph=False)
        pkg.lib().fppg_debug_fail_allocation(k)
        try:
            lose(b)
            break
        except pkg.FPPGError as e:
            assert e.code == pkg.ERR_OOM
        finally:
            pkg.lib().fppg_debug_fail_allocation(-1)
        n = held(b)
        if n == 500:                        # the failure came before its arrays were given up
            bt.store()
            continue
        assert n == 0
        for call in (bt.store, bt.load):
            with pytest.raises(pkg.FPPGError) as e:
                call()
            assert e.value.code == pkg.ERR_STATE
    assert k > 3


@pytest.mark.parametrize("replace", [lambda b: b.map_particles(), lose_by_setting])
def test_a_step_needs_the_forces_of_the_particles_it_moves(replace):
    b = body()
    amax = b.relax_forces()
    replace(b)
    with pytest.raises(pkg.FPPGError) as e:
        b.relax_step(amax)
    assert e.value.code == pkg.ERR_STATE
    b.relax_step(b.relax_forces())       # and then it goes on
