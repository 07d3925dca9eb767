"""hs_plan_info's device_bytes covers all that a plan holds, the second layout of its FP32
states included, while it is there."""

import pytest

from gpu_util import dev, make_plan, ragged_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("limited", [False, True])
@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_plan_info_counts_the_second_layout(cuda_device, prec, limited):
    import torch
    import __graft_entry__ as ge
    ge.build()
    from paper_1806_04596_gb300 import hypersara as hs
    c = ragged_case(n=64, L=3, M=(5000, 4000, 3000), seed=31)
    before = hs.device_bytes()
    try:
        hs.set_device_limit(1 << 40 if limited else 0)
        plan = make_plan(c, prec)
        alone = plan.info["device_bytes"]
        assert hs.device_bytes() == before + alone
        eps = torch.ones(3, dtype=torch.float64, device="cuda")
        st = hs.PDState(plan, dev(c["Y"], prec, True), eps, kappa3=1e-6, mu=0.01)
        first = plan.info["device_bytes"]
        held = hs.device_bytes()
        st2 = hs.PDState(plan, dev(c["Y"], prec, True), eps, kappa3=1e-6, mu=0.01)
        own = hs.device_bytes() - held            # of a state
        assert held == before + first + own
        assert first > alone if prec == "f32" else first == alone
        del st, st2
        assert hs.device_bytes() == before + plan.info["device_bytes"]
        assert plan.info["device_bytes"] == (alone if limited else first)
        del plan
        assert hs.device_bytes() == before
    finally:
        hs.set_device_limit(0)
