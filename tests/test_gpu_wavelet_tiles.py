"""Wavelet levels on 32 x 32 coefficient tiles (FP32, taken from two CTAs per SM on):
both directions against the FP64 oracle on images whose finest level, or finest two, use
them, with periodic wraps of 64-sample tiles, sides that are 3 or 5 times a power of
two, a single level, and caller buffers one element off an aligned address (bitwise equal to
the aligned result). Tolerances: the parity suite's."""

import numpy as np
import pytest

from gpu_util import assert_close, dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,L,levels", [(64, 64, 304, 1), (64, 64, 304, 4), (128, 64, 160, 2), (256, 128, 40, 3),
                                            (192, 128, 60, 2), (320, 64, 64, 2), (512, 512, 5, 4), (768, 256, 8, 3)])
def test_big_tiles_match_the_oracle(cuda_device, nx, ny, L, levels):
    import torch
    import __graft_entry__ as ge
    ge.build()
    from oracle import wavelets
    from paper_1806_04596_gb300 import hypersara as hs
    plan = hs.Plan(nx, ny, np.zeros(L + 1, dtype=np.int64), torch.zeros((0, 2), dtype=torch.float32, device="cuda"),
                   levels=levels, prec="f32", autotune=False)
    rng = np.random.Generator(np.random.PCG64(nx + 7 * ny + L))
    X = rng.standard_normal((L, ny, nx)).astype(np.float32)
    A = rng.standard_normal((9, L, ny, nx)).astype(np.float32)
    gA, gX = plan.psi_fwd(dev(X, "f32")), plan.psi_adj(dev(A, "f32"))
    ch = [0, L // 2, L - 1]
    a, x = host(gA)[:, ch], host(gX)[ch]
    assert_close(a, wavelets.psi_adjoint_cube(X[ch].astype(np.float64), levels), "f32")
    assert_close(x, wavelets.psi_cube(A[:, ch].astype(np.float64), levels), "f32")

    def off(t):
        b = torch.empty(t.numel() + 1, dtype=t.dtype, device="cuda")[1:].view(t.shape)
        b.copy_(t)
        return b

    oA = off(torch.empty_like(gA))
    plan.psi_fwd(off(dev(X, "f32")), oA)
    assert torch.equal(oA, gA)
    oX = off(torch.empty_like(gX))
    plan.psi_adj(off(dev(A, "f32")), oX)
    assert torch.equal(oX, gX)
