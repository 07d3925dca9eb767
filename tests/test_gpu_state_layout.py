"""The whole-plane layout that FP32 states with the nuclear prior iterate on, and the plan's
own half-plane calls beside it: both use the plan's grid, at different pitches."""

import time

import numpy as np
import pytest

from gpu_util import dev, make_plan, ragged_case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hs(cuda_device):
    import __graft_entry__ as ge
    ge.build()
    from paper_1806_04596_gb300 import hypersara
    return hypersara


def _case():
    return ragged_case(n=128, L=6, M=(60000, 50000, 0, 40000, 60000, 30000), seed=11)


def _state(hs, plan, c, **kw):
    import torch
    eps = torch.full((c["L"],), 5.0, dtype=torch.float64, device="cuda")
    return hs.PDState(plan, dev(c["Y"], plan.prec, True), eps, kappa3=1e-6, mu=0.01, **kw)


def test_later_states_take_the_layout_that_is_there(hs):
    """A state costs its own buffers (well under a millisecond); the layout, a quarter of a plan's
    work and more, is built once."""
    import torch
    c = _case()
    make_plan(c, "f32")                       # the tuner's choices of this shape
    torch.cuda.synchronize()
    t = time.perf_counter()
    plan = make_plan(c, "f32")
    torch.cuda.synchronize()
    t_plan = time.perf_counter() - t
    _state(hs, plan, c)
    ts = []
    for _ in range(5):
        torch.cuda.synchronize()
        t = time.perf_counter()
        st = _state(hs, plan, c)
        torch.cuda.synchronize()
        ts.append(time.perf_counter() - t)
        del st
    assert sorted(ts)[2] < 0.25 * t_plan, (ts, t_plan)
    before = hs.device_bytes()
    a = _state(hs, plan, c)
    one = hs.device_bytes() - before
    b = _state(hs, plan, c)
    assert hs.device_bytes() - before == 2 * one          # no layout among them
    del a, b
    assert hs.device_bytes() == before


@pytest.mark.parametrize("graph", [False, True])
def test_direct_calls_between_iterations(hs, graph):
    """Iterations between half-plane calls on the same plan are the bits of iterations alone, and
    the calls are the bits of calls alone."""
    import torch
    c = _case()
    plan = make_plan(c, "f32")
    X, Y = dev(c["X"], "f32"), dev(c["Y"], "f32", True)
    fwd, adj = plan.phi_fwd(X), plan.phi_adj(Y)
    st = _state(hs, plan, c)
    st.solve(6, graph)
    alone, beta, _ = st.get()
    alone = alone.clone()
    st = _state(hs, plan, c)
    for _ in range(3):
        st.solve(1, graph)
        assert torch.equal(plan.phi_fwd(X), fwd)
        st.solve(1, graph)
        assert torch.equal(plan.phi_adj(Y), adj)
    mixed, beta2, _ = st.get()
    assert torch.equal(mixed, alone) and beta2 == beta
    with_jas = _state(hs, plan, c, use_nuclear=False)    # iterates on the half plane
    with_jas.solve(4, graph)
    one = with_jas.get()[0].clone()
    both = _state(hs, plan, c, use_nuclear=False)
    st.set_data(Y, torch.full((c["L"],), 5.0, dtype=torch.float64, device="cuda"))
    for _ in range(4):
        both.solve(1, graph)
        st.solve(1, graph)
    assert torch.equal(both.get()[0], one)
