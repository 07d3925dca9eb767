"""Nuclear prox and singular values without a warm basis, over channel counts around every
padded size of the eigensolver (4, 8, 16, 32, 64): the parity suite's low-rank cube (a
rank-3 signal with small noise, graded weights), its reference (FP64 singular value
decomposition, the oracle's prox) and its tolerances, both forms, with few, no and all pairs
active, and a zero cube."""

import numpy as np
import pytest

from gpu_util import dev, host, rel
from oracle import prox

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dual", [False, True])
@pytest.mark.parametrize("L", [1, 4, 5, 8, 9, 16, 17, 32, 33, 60, 64])
def test_cold_nuclear_prox(cuda_device, L, dual):
    import torch
    import __graft_entry__ as ge
    ge.build()
    from paper_1806_04596_gb300 import hypersara as hs
    nx, ny = 64, 32
    plan = hs.Plan(nx, ny, np.zeros(L + 1, dtype=np.int64), torch.zeros((0, 2), dtype=torch.float32, device="cuda"),
                   levels=1, prec="f32", autotune=False)
    rng = np.random.default_rng(4 + L)
    S = rng.uniform(0, 1, (3, ny * nx))
    H = rng.uniform(0.5, 1.5, (L, 3))
    X = (H @ S + 0.01 * rng.standard_normal((L, ny * nx))).reshape(L, ny, nx).astype(np.float32).astype(np.float64)
    w = np.linspace(0.5, 1.5, L)
    ref_s = np.linalg.svd(X.reshape(L, -1).T, compute_uv=False)
    for thr in (2.0, 0.0, 1e4):
        out, sv = plan.prox_nuclear(dev(X, "f32"), thr, torch.tensor(w, dtype=torch.float64, device="cuda"), dual=dual)
        out, svh = host(out), host(sv)
        ref = prox.nuclear_dual(X, w, thr)[0] if dual else prox.prox_nuclear(X, w, thr)
        if np.linalg.norm(ref) > 0:
            assert rel(out, ref) <= 1e-5, (thr, rel(out, ref))
            assert np.max(np.abs(out - ref)) <= 1e-4 * np.max(np.abs(ref))
        else:
            assert np.all(np.abs(out) <= 1e-5 * np.max(np.abs(X)))
        act = ref_s > np.maximum(thr * w, 0.1) * 1.01
        act &= ref_s > 1e-2 * ref_s[0]   # the Gram matrix resolves sigma^2 to ~1e-7 sigma_max^2
        np.testing.assert_allclose(svh[act], ref_s[act], rtol=2e-6)
        assert np.max(np.abs(svh ** 2 - ref_s ** 2)) <= 4e-6 * ref_s[0] ** 2
    out, sv = plan.prox_nuclear(torch.zeros((L, ny, nx), dtype=torch.float32, device="cuda"), 0.5, dual=dual)
    assert torch.count_nonzero(out) == 0 and torch.count_nonzero(sv) == 0
    plan.check()
