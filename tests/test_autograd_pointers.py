"""Gradients that reach the kernels as bare pointers: what torch keeps beside the memory
(the conjugate and the negative bit) has to be in the memory, and a gradient that has no
memory (a batched one) must not get there. A stand-in plan on
the CPU reads every tensor the way the library does, from its address."""

import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1806_04596_gb300 import autograd as hsg


def _raw(t):
    """The tensor's memory, read through its address."""
    assert t.is_contiguous()
    n = t.numel() * (2 if t.is_complex() else 1)
    buf = (ctypes.c_double * n).from_address(t.data_ptr())
    a = np.array(buf[:], dtype=np.float64)
    return a.view(np.complex128).reshape(t.shape) if t.is_complex() else a.reshape(t.shape)


class _Plan:
    """Phi as a random L x ny x nx -> M matrix; the l2,1 norm and its direction as defined."""

    def __init__(self):
        rng = np.random.default_rng(5)
        self.F = rng.standard_normal((7, 12)) + 1j * rng.standard_normal((7, 12))

    def phi_fwd(self, X):
        return torch.tensor(self.F @ _raw(X).reshape(-1))

    def phi_adj(self, Y):
        return torch.tensor((self.F.conj().T @ _raw(Y)).real.reshape(3, 2, 2))

    def norm_l21(self, A, w_rows=None):
        return float(np.sqrt((_raw(A) ** 2).sum(axis=1)).sum())

    def l21_grad(self, A, w_rows=None, out=None, scale=None):
        a = _raw(A)
        g = a / np.sqrt((a ** 2).sum(axis=1, keepdims=True))
        return torch.tensor(g if scale is None else g * _raw(scale))


def test_negative_bit_of_the_incoming_gradient():
    plan = _Plan()
    A = torch.randn((9, 3, 2, 2), dtype=torch.float64, requires_grad=True)
    f = hsg.l21_norm(plan, A)
    (g1,) = torch.autograd.grad(f, A, retain_graph=True)
    z = torch.complex(torch.zeros_like(f), f).conj()        # -i f
    loss = (z * (2 + 3j)).real                               # 3 f, its gradient through a negated view
    (g3,) = torch.autograd.grad(loss, A, retain_graph=True)
    torch.testing.assert_close(g3, 3.0 * g1, rtol=1e-14, atol=0.0)


def test_conjugate_bit_of_the_incoming_gradient():
    plan = _Plan()
    X = torch.randn((3, 2, 2), dtype=torch.float64, requires_grad=True)
    w = torch.randn(7, dtype=torch.complex128)
    loss = (hsg.phi(plan, X).conj() * w).real.sum()
    (g,) = torch.autograd.grad(loss, X)
    want = (torch.tensor(plan.F.conj()) * w[:, None]).sum(0).real.reshape(3, 2, 2)
    torch.testing.assert_close(g, want, rtol=1e-13, atol=1e-13)


@pytest.mark.parametrize("vmapped", [False, True])
def test_batched_incoming_gradients(vmapped):
    plan = _Plan()
    A = torch.randn((9, 3, 2, 2), dtype=torch.float64, requires_grad=True)
    f = hsg.l21_norm(plan, A)
    (g1,) = torch.autograd.grad(f, A, retain_graph=True)
    c = torch.tensor([1.0, 2.0, -3.0], dtype=torch.float64)
    if vmapped:
        g = torch.vmap(lambda v: torch.autograd.grad(f, A, v, retain_graph=True)[0])(c)
    else:
        (g,) = torch.autograd.grad(f, A, grad_outputs=c, is_grads_batched=True, retain_graph=True)
    torch.testing.assert_close(g, c[:, None, None, None, None] * g1, rtol=1e-15, atol=0.0)
