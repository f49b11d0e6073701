"""Upstream gradients whose memory does not hold their value alone (a negative
bit, a forward-mode tangent) give the gradients that a torch scaling gives.  On
the CPU with a stand-in that reads the gradient's memory as the library does:
E = sum n^2 + sum (grad n)^3, dOmega = 1/4."""
import ctypes

import pytest

torch = pytest.importorskip("torch")
import torch.autograd.forward_ad as fwAD  # noqa: E402


class Stub:
    dOmega = 0.25

    def energy_gradients(self, n, grad, gE=None, E=None, dn=None, dg=None):
        if E is not None:
            E.copy_((n.double() ** 2).sum() + (grad.double() ** 3).sum())
        scale = None if gE is None else ctypes.c_double.from_address(gE.data_ptr()).value * self.dOmega
        if dn is not None:
            dn.copy_(8 * n * scale)
        if dg is not None:
            dg.copy_(12 * grad ** 2 * scale)

    def energy_potential(self, n, grad, E=None, v=None, w=None):
        v.copy_(8 * n)
        w.copy_(12 * grad ** 2)


@pytest.fixture
def energy():
    from paper_0812_0244_gb300.autograd import vdw_energy
    gen = torch.Generator().manual_seed(5)
    n = torch.rand(4, 5, 6, generator=gen, requires_grad=True)
    grad = torch.rand(3, 4, 5, 6, generator=gen, requires_grad=True)
    return n, grad, vdw_energy(n, grad, Stub())


def check(got, n, grad, scale):
    # a few FP32 roundings of products
    torch.testing.assert_close(got[0], 2 * n.detach() * scale, rtol=1e-6, atol=0)
    torch.testing.assert_close(got[1], 3 * grad.detach() ** 2 * scale, rtol=1e-6, atol=0)


@pytest.mark.parametrize("kind", ["plain", "expanded", "offset", "neg_view", "imag_of_conj", "zero"])
def test_memory_and_value(energy, kind):
    n, grad, E = energy
    base = torch.tensor([0.5, -1.75, 3.0], dtype=torch.float64)
    gE = {
        "plain": lambda: base[1].clone(),
        "expanded": lambda: base[1:2].expand(2)[1],
        "offset": lambda: base[1],
        "neg_view": lambda: torch._neg_view(base[1]),
        "imag_of_conj": lambda: torch.complex(base, base).conj().imag[1],
        "zero": lambda: torch._efficientzerotensor((), dtype=torch.float64),
    }[kind]()
    scale = {"neg_view": 1.75, "imag_of_conj": 1.75, "zero": 0.0}.get(kind, -1.75)
    check(torch.autograd.grad(E, (n, grad), grad_outputs=gE), n, grad, scale)


def test_negative_bit_from_a_complex_loss(energy):
    """The upstream gradient that autograd itself makes."""
    n, grad, E = energy
    loss = (torch.complex(torch.zeros_like(E), E).conj() * (2.0 + 3.0j)).real  # 3 E
    check(torch.autograd.grad(loss, (n, grad)), n, grad, 3.0)


def test_tangent_of_the_upstream_gradient(energy):
    n, grad, E = energy
    with fwAD.dual_level():
        gE = fwAD.make_dual(torch.tensor(2.0, dtype=torch.float64), torch.tensor(-0.5, dtype=torch.float64))
        got = [fwAD.unpack_dual(t) for t in torch.autograd.grad(E, (n, grad), grad_outputs=gE)]
        assert all(t.tangent is not None for t in got)
        check([t.primal for t in got], n, grad, 2.0)
        check([t.tangent for t in got], n, grad, -0.5)
