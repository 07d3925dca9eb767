"""l2,1 norm of FP32 cubes with weights of exactly zero among others: masked rows leave
nothing (also -0), masked rows that are not finite leave NaN, as 0 * inf does. Rows carry
FP64 accuracy, so 1e-14 holds with room."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [1, 5, 20])
def test_norm_l21_with_masked_rows(cuda_device, L):
    import torch
    import __graft_entry__ as ge
    ge.build()
    from paper_1806_04596_gb300 import hypersara as hs
    plan = hs.Plan(32, 16, np.zeros(L + 1, dtype=np.int64), torch.zeros((0, 2), dtype=torch.float32, device="cuda"),
                   levels=1, prec="f32", autotune=False)
    rng = np.random.Generator(np.random.PCG64(L))
    A = rng.standard_normal((9, L, 512)).astype(np.float32)
    A[3] *= np.float32(1e-30)
    A[4, :, 7] = 0.0
    w = np.where(rng.uniform(size=(9, 512)) < 0.5, 0.0, rng.uniform(size=(9, 512))).astype(np.float32)
    w[1, ::2] = -0.0
    w[2, 3] = 0.0
    t = torch.tensor(A, device="cuda")
    want = float((np.sqrt(np.sum(A.astype(np.float64) ** 2, axis=1)) * w).sum())
    assert abs(plan.norm_l21(t, torch.tensor(w, device="cuda")) - want) <= 1e-14 * want
    assert plan.norm_l21(t, torch.zeros((9, 16, 32), device="cuda")) == 0.0
    for bad in (np.inf, np.nan):
        t[2, 0, 3] = bad
        assert np.isnan(plan.norm_l21(t, torch.tensor(w, device="cuda")))
