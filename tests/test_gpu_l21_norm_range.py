"""l2,1 norm of FP32 cubes where the products of rows and weights lie near the ends of the
FP32 range, over enough rows that a thread adds many of them: finite inputs give the
finite sum. Rows are equal, so the sum is rows x root x weight; a thread adds at most
42 rows at this size and the sums after it are trees of 18 levels, so 1e-14 holds with
room."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("coef,weight", [(1.9 * 2.0 ** 62, 2.0 ** 60), (2.0 ** 62, -(2.0 ** 59)), (1.5 * 2.0 ** 62, 1.0),
                                         (3e38, 2.5e38), (1e-12, 1e-30), (1e-30, 1e-38)])
def test_norm_l21_near_the_ends_of_the_range(cuda_device, coef, weight):
    import torch
    import __graft_entry__ as ge
    ge.build()
    from paper_1806_04596_gb300 import hypersara as hs
    n = 1024
    plan = hs.Plan(n, n, np.zeros(2, dtype=np.int64), torch.zeros((0, 2), dtype=torch.float32, device="cuda"),
                   levels=1, prec="f32", autotune=False)
    A = torch.full((9, 1, n, n), coef, dtype=torch.float32, device="cuda")
    w = torch.full((9, n, n), weight, dtype=torch.float32, device="cuda")
    want = 9.0 * n * n * float(np.float32(coef)) * float(np.float32(weight))
    assert abs(plan.norm_l21(A, w) - want) <= 1e-14 * abs(want)
    w[8, -1, -1] = np.inf
    assert plan.norm_l21(A, w) == np.inf
