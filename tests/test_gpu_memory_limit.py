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
