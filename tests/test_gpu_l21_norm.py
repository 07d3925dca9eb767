"""FP32 l2,1 norm by exact square pairs: against FP64 sums over channel counts around
the four-warp split, with rows that leave the pairs' range (huge, tiny, zero, infinite)
and an unaligned buffer (the plain form). A row's pair sum carries 46 bits and rows add
in FP64, so 1e-13 relative holds with room. The scaled direction equals the direction
times the factor bit for bit."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _plan(L):
    import torch
    import __graft_entry__ as ge
    ge.build()
    from paper_1806_04596_gb300 import hypersara as hs
    off = np.arange(L + 1, dtype=np.int64)
    return hs.Plan(32, 16, off, torch.zeros((L, 2), dtype=torch.float32, device="cuda"), levels=1, prec="f32",
                   autotune=False)


@pytest.mark.parametrize("unaligned", [False, True])
@pytest.mark.parametrize("weights", [False, True])
@pytest.mark.parametrize("L", [1, 3, 4, 33, 64, 70])
def test_norm_l21_over_the_fp32_range(cuda_device, L, weights, unaligned):
    import torch
    plan = _plan(L)
    rng = np.random.Generator(np.random.PCG64(L))
    A = rng.standard_normal((9, L, 512)) * 10.0 ** rng.uniform(-3, 3, (9, 1, 512))
    A[0, :, :64] = 0.0
    A[1, :, 5] *= 1e25          # squares overflow FP32
    A[2, :, 7] *= 1e-25         # squares underflow
    A[3, :, 9] = 1e-38
    A[4, 0, 11] = 3e38
    A[5, :, 100:200] *= 1e-12
    A = A.astype(np.float32)
    w = rng.uniform(0.0, 1.0, (9, 512)).astype(np.float32) if weights else None
    t = torch.empty(A.size + 1, dtype=torch.float32, device="cuda")[1 if unaligned else 0:][:A.size]
    t.copy_(torch.tensor(A.reshape(-1)))
    wt = None if w is None else torch.tensor(w.reshape(-1), device="cuda")

    def ref(a):
        n = np.sqrt(np.sum(a.astype(np.float64) ** 2, axis=1))
        return n if w is None else n * w.astype(np.float64)

    assert abs(plan.norm_l21(t, wt) - ref(A).sum()) <= 1e-13 * ref(A).sum()
    A[1, :, 5] = A[4, :, 11] = 0.0   # without the rows that swamp the sum
    t.copy_(torch.tensor(A.reshape(-1)))
    assert abs(plan.norm_l21(t, wt) - ref(A).sum()) <= 1e-13 * ref(A).sum()
    if not weights:
        A[6, 0, 1] = np.inf
        t.copy_(torch.tensor(A.reshape(-1)))
        assert plan.norm_l21(t) == np.inf
        A[6, 0, 1] = np.nan
        t.copy_(torch.tensor(A.reshape(-1)))
        assert np.isnan(plan.norm_l21(t))


@pytest.mark.parametrize("prec,L", [("f32", 3), ("f32", 64), ("f32", 70), ("f64", 5)])
def test_scaled_direction_is_the_product(cuda_device, prec, L):
    import torch
    import __graft_entry__ as ge
    ge.build()
    from paper_1806_04596_gb300 import hypersara as hs
    rdt = torch.float32 if prec == "f32" else torch.float64
    plan = hs.Plan(32, 16, np.arange(L + 1, dtype=np.int64), torch.zeros((L, 2), dtype=rdt, device="cuda"), levels=1,
                   prec=prec, autotune=False)
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    A = torch.randn((9, L, 16, 32), generator=g, dtype=rdt, device="cuda")
    A[0, :, 0, 0] = 0
    for v in (0.37, -2.5, float("inf")):
        s = torch.tensor(v, dtype=rdt, device="cuda")
        want, got = plan.l21_grad(A) * s, plan.l21_grad(A, scale=s)
        assert torch.equal(torch.nan_to_num(want, nan=7.0), torch.nan_to_num(got, nan=7.0))
    with pytest.raises(ValueError):
        plan.l21_grad(A, scale=torch.ones(2, dtype=rdt, device="cuda"))
