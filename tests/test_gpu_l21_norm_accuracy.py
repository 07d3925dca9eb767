"""l2,1 norm of FP32 cubes to FP64 accuracy: the mean relative error over 16 cubes against
extended precision (64 bits or more). A sum rounded at every level of its tree has its
error from the last levels, 2^-54 / sqrt 3 in the last one and half of that variance in each before:
6e-17 in root mean square when every row is right to FP64. Rows that carry fewer bits
(46 to 48) or are added in fewer show as 2e-16 and more. Bound on the mean: 2^-53."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,L", [(16, 16, 1), (64, 64, 8), (96, 160, 5), (64, 64, 60), (32, 64, 70)])
def test_norm_l21_is_as_accurate_as_fp64_sums(cuda_device, nx, ny, L):
    import torch
    import __graft_entry__ as ge
    ge.build()
    from paper_1806_04596_gb300 import hypersara as hs
    plan = hs.Plan(nx, ny, np.zeros(L + 1, dtype=np.int64), torch.zeros((0, 2), dtype=torch.float32, device="cuda"),
                   levels=1, prec="f32", autotune=False)
    ext = np.longdouble
    errs = []
    for seed in range(16):
        rng = np.random.Generator(np.random.PCG64(seed))
        A = (rng.standard_normal((9, L, ny * nx)) * rng.standard_normal((9, 1, ny * nx))).astype(np.float32)
        n2 = np.zeros((9, ny * nx), dtype=ext)
        for l in range(L):
            n2 += A[:, l].astype(ext) ** 2
        want = np.sqrt(n2).sum()
        got = plan.norm_l21(torch.tensor(A.reshape(9, L, ny, nx), device="cuda"))
        errs.append(float(abs(ext(got) - want) / want))
    assert np.mean(errs) <= 2.0 ** -53, errs
