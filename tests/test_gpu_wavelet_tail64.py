"""FP64 wavelet levels whose shared-memory tail starts at 32 samples when the tails are
few, and at 64 when they are many: both directions against the FP64 oracle on
either side of that line, on squares and oblongs, with one to two levels in the tail.
Tolerances: the parity suite's."""

import numpy as np
import pytest

from gpu_util import assert_close, dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [1, 7, 15, 16, 20])
@pytest.mark.parametrize("nx,ny,levels", [(64, 64, 2), (128, 128, 2), (128, 128, 3), (128, 64, 2), (128, 256, 3), (256, 128, 3)])
def test_fp64_tails_match_the_oracle(cuda_device, nx, ny, levels, L):
    import torch
    import __graft_entry__ as ge
    ge.build()
    from oracle import wavelets
    from paper_1806_04596_gb300 import hypersara as hs
    plan = hs.Plan(nx, ny, np.zeros(L + 1, dtype=np.int64), torch.zeros((0, 2), dtype=torch.float64, device="cuda"),
                   levels=levels, prec="f64", autotune=False)
    rng = np.random.Generator(np.random.PCG64(nx + 7 * ny + L))
    X = rng.standard_normal((L, ny, nx))
    A = rng.standard_normal((9, L, ny, nx))
    ch = sorted({0, L // 2, L - 1})
    assert_close(host(plan.psi_fwd(dev(X, "f64")))[:, ch], wavelets.psi_adjoint_cube(X[ch], levels), "f64")
    assert_close(host(plan.psi_adj(dev(A, "f64")))[ch], wavelets.psi_cube(A[:, ch], levels), "f64")
