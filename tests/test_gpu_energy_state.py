"""The energy's forward leaves the gradients to the backward: it does none of
their work, and what it leaves gives the gradients of its own moment, whatever
happens to the body before they are asked for."""
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


def body(odd=0):
    a = W.cube_workload(seed=4)[0]
    b = pkg.Body(a.verts, a.tris, a.dx, a.h)
    b.extract_features(a.dihedral_deg)
    keep = slice(0, len(a.xyz) - (len(a.xyz) + odd) % 2)
    b.set_particles(a.xyz[keep], a.cls[keep])
    b.relax(2)
    return b


def inputs(b):
    import torch
    y = torch.from_numpy(b.get_particles()[0]).cuda().requires_grad_(True)
    return y, torch.from_numpy(b.verts).cuda().requires_grad_(True)


def reference(b, y, v):
    import torch
    gy, gv = torch.empty_like(y), torch.empty_like(v)
    E = b.energy_ptr(y.data_ptr(), v.data_ptr(), gy.data_ptr(), gv.data_ptr())
    torch.cuda.synchronize()
    return E, gy.detach(), gv.detach()


def test_a_forward_alone_does_no_work_of_the_backward():
    # with the gradients in it a forward took five times as long as without
    import time

    import torch
    from paper_2501_03056_gb300.autograd import uniformity_energy
    b = body()
    y, v = inputs(b)

    def took(f):
        runs = []
        for _ in range(25):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            f()
            torch.cuda.synchronize()
            runs.append(time.perf_counter() - t0)
        return sorted(runs)[12]

    with torch.no_grad():
        alone = took(lambda: uniformity_energy(y, v, b))
    assert took(lambda: uniformity_energy(y, v, b)) < 2.0 * alone


def new_particles(b):
    b.set_particles(np.zeros((17, 3), np.float32), np.full(17, W.CLS_V, np.int32))


@pytest.mark.parametrize("between", [
    lambda b: None, lambda b: b.relax(5), new_particles, lambda b: b.map_particles(),
    lambda b: b.set_cell_order(pkg.ORDER_MORTON_ROWS), lambda b: b.set_cell_order(pkg.ORDER_ROWS),
    lambda b: b.set_mobile_classes((W.CLS_S,)), lambda b: b.set_incremental(False)])
@pytest.mark.parametrize("counted,order,odd", [
    (True, pkg.ORDER_ROWS, 0), (True, pkg.ORDER_MORTON_ROWS, 1), (False, pkg.ORDER_ROWS, 1),
    (False, pkg.ORDER_MORTON_ROWS, 0)])
def test_the_gradients_are_those_of_the_forward(between, counted, order, odd):
    import torch
    from paper_2501_03056_gb300.autograd import uniformity_energy
    b = body(odd)
    b.set_incremental(counted)
    b.set_cell_order(order)
    y, v = inputs(b)
    E, gy, gv = reference(b, y, v)
    e = uniformity_energy(y, v, b)
    assert float(e.detach()) == E
    between(b)
    got = torch.autograd.grad(e, (y, v))
    assert torch.equal(got[0], gy) and torch.equal(got[1], gv)


def test_a_forward_leaves_a_split_iteration_alone():
    import torch
    from paper_2501_03056_gb300.autograd import uniformity_energy
    a, b = body(), body()
    y, v = inputs(b)
    for q in (a, b):
        amax = q.relax_forces()
        if q is b:
            torch.autograd.grad(uniformity_energy(y + 0.01, v, q), y)
        q.relax_step(amax)
    assert all(np.array_equal(p, q) for p, q in zip(a.get_particles(), b.get_particles()))


def test_streams_and_moved_states():
    # backwards still under way on one stream, the next forward on another;
    # a state that went through host memory
    import torch
    from paper_2501_03056_gb300.autograd import uniformity_energy
    b = body()
    y, v = inputs(b)
    E, gy, gv = reference(b, y, v)
    streams = [torch.cuda.Stream() for _ in range(2)]
    got = []
    torch.cuda.synchronize()
    for k in range(8):
        with torch.cuda.stream(streams[k % 2]):
            e = uniformity_energy(y, v, b)
            got.append((e.detach(), *torch.autograd.grad(e, (y, v))))
    with torch.autograd.graph.save_on_cpu():
        e = uniformity_energy(y, v, b)
    got.append((e.detach(), *torch.autograd.grad(e, (y, v))))
    torch.cuda.synchronize()
    for e, a, c in got:
        assert float(e) == E and torch.equal(a, gy) and torch.equal(c, gv)


def test_bad_states_and_failed_allocations_are_refused():
    import torch
    b = body()
    y, v = inputs(b)
    size = b.energy_state_bytes(b.n)
    assert size >= 48 * b.n and b.energy_state_bytes(-1) == -1
    state = torch.empty(size + 16, dtype=torch.uint8, device="cuda")
    gy, gv = torch.empty_like(y), torch.empty_like(v)
    for ptr, n in ((0, size), (state.data_ptr() + 4, size), (state.data_ptr(), size - 1)):
        for call in (lambda: b.energy_forward_ptr(y.data_ptr(), v.data_ptr(), ptr, n),
                     lambda: b.energy_backward_ptr(b.n, y.data_ptr(), v.data_ptr(), ptr, n, gy.data_ptr())):
            with pytest.raises(pkg.FPPGError) as e:
                call()
            assert e.value.code == pkg.ERR_ARG
    k = 0
    while True:
        fresh = body()
        pkg.lib().fppg_debug_fail_allocation(k)
        try:
            E = fresh.energy_forward_ptr(y.data_ptr(), v.data_ptr(), state.data_ptr(), size)
            break
        except pkg.FPPGError as e:
            assert e.code == pkg.ERR_OOM
            k += 1
        finally:
            pkg.lib().fppg_debug_fail_allocation(-1)
    assert k > 5 and E == reference(b, y, v)[0]
    # no particles: no energy, and vertex gradients of zero
    b.set_particles(np.zeros((0, 3), np.float32), np.zeros(0, np.int32))
    assert b.energy_forward_ptr(y.data_ptr(), v.data_ptr(), 0, 0) == 0.0
    gv.detach().fill_(1.0)
    b.energy_backward_ptr(0, 0, v.data_ptr(), 0, 0, 0, gv.data_ptr())
    torch.cuda.synchronize()
    assert not gv.detach().any()
    assert pkg.lib().fppg_energy_forward(None, None, None, ctypes.byref(ctypes.c_double()), None, 0) == pkg.ERR_ARG
