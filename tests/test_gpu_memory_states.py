"""Several solver states under hs_set_device_limit: as many FP32 states with the nuclear prior, and
their staging for host data, fit beside a plan as would beside one set of lists and wavelet
scratch of two coefficient cubes, at sparse and at dense coverage (in between the first state's second layout
would fit in the room of the second state)."""

import numpy as np
import pytest

from gpu_util import dev, host, make_plan, ragged_case, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M", [(2000, 1503, 0, 911), (20000, 15000, 20000, 0), (60000, 40000, 50000, 0)])
def test_two_states_and_host_data_fit_under_a_limit(cuda_device, M):
    import torch
    import __graft_entry__ as ge
    ge.build()
    from paper_1806_04596_gb300 import hypersara as hs
    c = ragged_case(n=64, L=4, M=M, seed=24)
    n, m = 64 * 64 * 4, int(c["off"][-1])
    Y = dev(c["Y"], "f32", True)
    eps = torch.full((4,), 5.0, dtype=torch.float64, device="cuda")

    def state(plan, **kw):
        return hs.PDState(plan, Y, eps, kappa3=1e-6, mu=0.01, **kw)

    plan = make_plan(c, "f32")
    held = hs.device_bytes()
    jas = state(plan, use_nuclear=False)
    one = hs.device_bytes() - held   # a state without a layout of its own
    del jas
    scratch = 2 * 8 * (n - n // 4) * 4   # of two coefficient cubes, beside what the plan holds
    before = hs.device_bytes()
    try:
        hs.set_device_limit(before + scratch + 2 * one + 8 * m)
        a = state(plan)
        b = state(plan)
        Yh, eh = Y.cpu().pin_memory(), eps.cpu().numpy()
        a.set_data_host(Yh, eh)
        for st in (a, b):
            st.solve(3, graph=True)
        assert rel(host(a.get()[0]), host(b.get()[0])) == 0.0   # one layout for both
        assert np.isfinite(a.get()[1])
    finally:
        hs.set_device_limit(0)
