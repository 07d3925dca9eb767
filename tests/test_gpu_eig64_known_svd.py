"""FP64 nuclear prox of cubes whose singular value decomposition is exact: X = H diag(s) W^T
with rows of Walsh-Hadamard matrices (entries +- a power of two) and singular values of a few
bits, so that X and its soft threshold are exact in FP64. A column of the eigenvectors meets
at most nine sweeps of L - 1 rotations, each rounded to 2^-53: as errors of either sign they add to
sqrt(9 (L - 1)) 2^-53. The bound is twice that; rotations that are off the unit circle to
one side add up to (9 (L - 1)) 2^-53 instead."""

import numpy as np
import pytest

from gpu_util import dev, host

pytestmark = pytest.mark.gpu


def _hadamard(n):
    h = np.ones((1, 1))
    while len(h) < n:
        h = np.block([[h, h], [h, -h]])
    return h


@pytest.mark.parametrize("dual", [False, True])
@pytest.mark.parametrize("L", [4, 16, 64])
def test_fp64_nuclear_prox_of_a_known_decomposition(cuda_device, L, dual):
    import torch
    import __graft_entry__ as ge
    ge.build()
    from paper_1806_04596_gb300 import hypersara as hs
    nx = ny = 32
    plan = hs.Plan(nx, ny, np.zeros(L + 1, dtype=np.int64), torch.zeros((0, 2), dtype=torch.float64, device="cuda"),
                   levels=1, prec="f64", autotune=False)
    rng = np.random.default_rng(L)
    g = int(np.log2(L))
    H = _hadamard(L) * 2.0 ** -(g // 2)                     # g even: orthogonal to the bit
    W = _hadamard(nx * ny)[rng.permutation(nx * ny)[:L]] / 32.0
    s = np.concatenate([[1024.0, 640.0, 384.0], (8 + rng.permutation(L - 3)) / 16.0])
    thr = 32.0
    X = (H * s) @ W
    f = np.minimum(s, thr) if dual else np.maximum(s - thr, 0.0)
    want = (H * f) @ W
    out, sv = plan.prox_nuclear(dev(X.reshape(L, ny, nx), "f64"), thr, dual=dual)
    err = np.linalg.norm(host(out).reshape(L, -1) - want) / np.linalg.norm(X if dual else want)
    assert err <= 2.0 * np.sqrt(9.0 * (L - 1)) * 2.0 ** -53, err
    np.testing.assert_allclose(host(sv)[:3], s[:3], rtol=1e-13)
