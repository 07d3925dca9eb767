"""Plans and solver states under hs_set_device_limit: what fits with one whole-plane grid, one
set of lists and no tables still fits, and gives the same results."""

import numpy as np
import pytest

from gpu_util import TOL, dev, host, make_plan, oracle_op, ragged_case, rel

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hs(cuda_device):
    import __graft_entry__ as ge
    ge.build()
    from paper_1806_04596_gb300 import hypersara
    return hypersara


def _state(hs, plan, c, **kw):
    import torch
    eps = torch.full((c["L"],), 5.0, dtype=torch.float64, device="cuda")
    return hs.PDState(plan, dev(c["Y"], plan.prec, True), eps, kappa3=1e-6, mu=0.01, **kw)


def _state_bytes(c, r):
    """A state's cubes and visibility vectors and, per block, its sums (generously)."""
    n, M = c["L"] * c["ny"] * c["nx"], int(c["off"][-1])
    return r * (23 * n + 6 * M) + (1 << 20)


@pytest.mark.parametrize("M", [(2000, 1503, 0, 911), (60000, 40000, 50000, 0)])
def test_fp64_tables_leave_the_states_room(hs, M):
    """Sparse and dense coverage: under a limit a plan holds at most what it would without the tables
    (128 bytes a visibility) and with the grid scratch of the whole plane (K x K and n x K complex
    values a channel instead of K x 96 and (n + 8) x K), so that a state still fits."""
    c = ragged_case(n=64, L=4, M=M, seed=21)
    n, K, L, m = 64, 128, 4, int(c["off"][-1])
    free = make_plan(c, "f64")
    want = host(free.phi_adj(dev(c["Y"], "f64", True)))
    with_tables = free.info["device_bytes"]
    del free
    before = hs.device_bytes()
    whole = with_tables - 128 * m + L * 16 * (K * (K - 96) + n * (K - n - 8))   # no tables, whole plane
    try:
        hs.set_device_limit(before + whole + _state_bytes(c, 8))
        plan = make_plan(c, "f64")
        assert plan.info["device_bytes"] <= whole
        st = _state(hs, plan, c)
        st.solve(3, graph=False)
        X, beta, rho = st.get()
        assert np.isfinite(beta)
        assert rel(host(plan.phi_adj(dev(c["Y"], "f64", True))), want) <= TOL["f64"]
        assert rel(host(plan.phi_fwd(dev(c["X"], "f64"))), oracle_op(c).forward(c["X"])) <= TOL["f64"]
    finally:
        hs.set_device_limit(0)


@pytest.mark.parametrize("M", [(2000, 1503, 0, 911), (60000, 40000, 50000, 0)])
def test_fp32_states_fit_beside_one_set_of_lists(hs, M):
    """A state with the nuclear prior where the limit leaves room for the state alone: it
    iterates without a second layout, to the iterates of a state that has one (FP32 sums
    in another order: 1e-5 an operator, which the warm-started eigensolver turns into at most
    4e-4 of the image in ten iterations; three here)."""
    c = ragged_case(n=64, L=4, M=M, seed=22)
    plan = make_plan(c, "f32")
    free = _state(hs, plan, c)
    free.solve(3, graph=False)
    want = host(free.get()[0])
    del free, plan
    plan = make_plan(c, "f32")
    jas = _state(hs, plan, c, use_nuclear=False)
    before = hs.device_bytes()
    jas2 = _state(hs, plan, c, use_nuclear=False)
    one = hs.device_bytes() - before
    del jas, jas2
    before = hs.device_bytes()
    try:
        hs.set_device_limit(before + one)
        st = _state(hs, plan, c)
        assert hs.device_bytes() <= before + one
        st.solve(3, graph=True)
        assert rel(host(st.get()[0]), want) <= 1e-4
        hs.set_device_limit(before + one - 4096)
        with pytest.raises(hs.HSError) as e:
            _state(hs, plan, c)
        assert e.value.status == hs.HS_ERR_NOMEM
        assert hs.device_bytes() == before + one       # nothing left of the attempt
    finally:
        hs.set_device_limit(0)


@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_plan_and_state_hold_no_more_than_with_one_layout(hs, prec):
    """At a visibility and a half per pixel and channel, the bytes of a plan with the whole
    plane's grid, one set of lists (24 bytes a visibility, 40 in FP64) and wavelet scratch of two
    coefficient cubes."""
    n, L = 128, 8
    m = 3 * n * n // 2
    c = ragged_case(n=n, L=L, M=(m,) * L, seed=23)
    r = 4 if prec == "f32" else 8
    K = 2 * n
    before = hs.device_bytes()
    try:
        hs.set_device_limit(1 << 40)
        plan = make_plan(c, prec)
        st = _state(hs, plan, c)
        N = n * n * L
        whole = 2 * r * L * (K * K + n * K) + r * (16 + 2) * N + (2 * r + 8 + 4 * r) * m * L + (1 << 20)
        assert hs.device_bytes() - before <= whole + _state_bytes(c, r)
        del st
    finally:
        hs.set_device_limit(0)
