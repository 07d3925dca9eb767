"""Nuclear prox and singular values without a warm basis do not depend on the units of the
cube: times a power of two (threshold too) they are the same bits times that power, up to
cubes whose Gram matrix has squares beyond the FP32 range and down to those whose squares vanish in it."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dual", [False, True])
@pytest.mark.parametrize("L", [5, 8, 17, 60, 64])
def test_cold_nuclear_prox_scales_exactly(cuda_device, L, dual):
    import torch
    import __graft_entry__ as ge
    ge.build()
    from paper_1806_04596_gb300 import hypersara as hs
    nx, ny = 64, 32
    plan = hs.Plan(nx, ny, np.zeros(L + 1, dtype=np.int64), torch.zeros((0, 2), dtype=torch.float32, device="cuda"),
                   levels=1, prec="f32", autotune=False)
    rng = np.random.default_rng(L)
    X = rng.uniform(0.5, 1.5, (L, 3)) @ rng.uniform(0, 1, (3, nx * ny)) + 0.01 * rng.standard_normal((L, nx * ny))
    X = torch.tensor(X.reshape(L, ny, nx), dtype=torch.float32, device="cuda")
    out, sv = plan.prox_nuclear(X, 2.0, dual=dual)
    for k in (18, 22, 23, 24, 26, 30, 45, -20, -30, -45):
        f = 2.0 ** k
        o, s = plan.prox_nuclear(X * f, 2.0 * f, dual=dual)
        assert torch.equal(o, out * f) and torch.equal(s, sv * f), k
    plan.check()
