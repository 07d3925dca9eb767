"""Half-plane measurement operator: samples with u < 0 are mirrored to (-u, -v)
and conjugated, so the edges of the half plane and samples on grid cells are
where it could go wrong. Both directions against the FP64 oracle on coverage
made of cell points (integer t = u K / (2 pi), where the window's tie-break
acts), axis points (u = 0, v = 0), points within one window of both ends of the
u axis, and random ones, over the line lengths of every FFT form (2^a, 3 2^a,
5 2^a) and non-square images. Tolerances: the parity suite's."""

import numpy as np
import pytest

from gpu_util import assert_close, dev, host, oracle_op, rounded

pytestmark = pytest.mark.gpu

SHAPES = [(16, 16), (16, 64), (32, 16), (64, 32), (96, 32), (32, 160), (128, 192), (320, 64), (64, 768),
          (1024, 16), (16, 1280), (640, 96)]


def _edge_case(nx, ny, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    Kx, Ky = 2 * nx, 2 * ny
    cells = np.stack([rng.integers(-Kx // 2, Kx // 2, 60), rng.integers(-Ky // 2, Ky // 2, 60)], axis=1)
    axes = np.array([[0, 0], [0, 3], [0, -3], [5, 0], [-5, 0], [-1, 0], [-1, -1], [1, -1], [-Kx // 2, 1],
                     [-Kx // 2, -Ky // 2], [Kx // 2 - 1, Ky // 2 - 1], [-Kx // 2 + 1, -1]])
    t = np.concatenate([cells, axes]).astype(np.float64)
    near = np.concatenate([rng.uniform(-4.5, 4.5, 40), Kx / 2 - rng.uniform(0.0, 4.5, 20),
                           -Kx / 2 + rng.uniform(0.0, 4.5, 20)])
    t = np.concatenate([t, np.stack([near, rng.uniform(-Ky / 2, Ky / 2, near.size)], axis=1),
                        np.stack([rng.uniform(-Kx / 2, Kx / 2, 90), rng.uniform(-Ky / 2, Ky / 2, 90)], axis=1)])
    uv = np.clip(t * 2.0 * np.pi / np.array([Kx, Ky]), -np.pi, np.nextafter(np.pi, 0.0))
    off = np.array([0, 100, 100, len(uv)], dtype=np.int64)   # an empty channel between
    X = rng.uniform(-0.5, 1.0, (3, ny, nx))
    Y = rng.standard_normal(len(uv)) + 1j * rng.standard_normal(len(uv))
    return dict(nx=nx, ny=ny, L=3, off=off, uv=uv, X=X, Y=Y, rng=rng)


@pytest.mark.parametrize("compensated", [False, True])
@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("nx,ny", SHAPES)
def test_edges_of_the_half_plane_match_the_oracle(cuda_device, nx, ny, prec, compensated):
    import __graft_entry__ as ge
    ge.build()
    from paper_1806_04596_gb300 import hypersara as hs
    c = _edge_case(nx, ny, seed=nx * 7919 + ny)
    if prec == "f32":   # FP32 radians inside [-pi, pi) as FP64 compares them
        lim = np.nextafter(np.float32(np.pi), np.float32(0.0))
        c["uv"] = np.clip(c["uv"].astype(np.float32), -lim, lim).astype(np.float64)
    c = rounded(c, prec)
    plan = hs.Plan(nx, ny, c["off"], dev(c["uv"], prec), levels=1, prec=prec, compensated=compensated)
    op = oracle_op(c)
    assert_close(host(plan.phi_fwd(dev(c["X"], prec))), op.forward(c["X"]), prec)
    assert_close(host(plan.phi_adj(dev(c["Y"], prec, True))), op.adjoint(c["Y"]), prec)


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("nx,ny,M", [(32, 32, 1), (32, 96, 33), (64, 64, 4000), (96, 64, 2500), (64, 320, 3000)])
def test_shared_gridding_items_match_the_oracle(cuda_device, nx, ny, M, prec):
    """Few, dense work items, where the tuner takes the form with several warps to
    an item: one window, one batch and a bit, and thousands of windows packed into a
    few rows around the origin (so that every warp of an item holds a share)."""
    import __graft_entry__ as ge
    ge.build()
    from paper_1806_04596_gb300 import hypersara as hs
    rng = np.random.Generator(np.random.PCG64(1000 * nx + ny + M))
    uv = rng.normal(0.0, [16.0 * np.pi / nx, 10.0 * np.pi / ny], (2 * M, 2))
    uv = np.clip(uv, -3.0, 3.0)
    c = dict(nx=nx, ny=ny, L=2, off=np.array([0, M, 2 * M], dtype=np.int64), uv=uv, X=np.zeros((2, ny, nx)),
             Y=rng.standard_normal(2 * M) + 1j * rng.standard_normal(2 * M), rng=rng)
    c = rounded(c, prec)
    plan = hs.Plan(nx, ny, c["off"], dev(c["uv"], prec), levels=1, prec=prec)
    assert_close(host(plan.phi_adj(dev(c["Y"], prec, True))), oracle_op(c).adjoint(c["Y"]), prec)
