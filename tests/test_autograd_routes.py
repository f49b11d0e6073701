"""The backward's two routes (scaling by the upstream gradient inside the
assembly kernel, or as a torch operation) give the same gradients, on the CPU
with a stand-in for the library: E = sum n^2 + sum (grad n)^3, dOmega = 1/4."""
import pytest


class Stub:
    dOmega = 0.25

    def energy_gradients(self, n, grad, gE=None, E=None, dn=None, dg=None):
        for t in (n, grad, gE, E, dn, dg):
            assert t is None or t.data_ptr()  # as the library takes them
        if E is not None:
            E.copy_((n.double() ** 2).sum() + (grad.double() ** 3).sum())
        scale = None if gE is None else (gE * self.dOmega).float()
        if dn is not None:
            dn.copy_(8 * n * scale)
        if dg is not None:
            dg.copy_(12 * grad ** 2 * scale)

    def energy_potential(self, n, grad, E=None, v=None, w=None):
        assert n.data_ptr() and grad.data_ptr()
        v.copy_(8 * n)
        w.copy_(12 * grad ** 2)


@pytest.mark.parametrize("route", ["plain", "create_graph", "batched"])
@pytest.mark.parametrize("wants", ["both", "n", "grad"])
def test_routes_agree(route, wants):
    torch = pytest.importorskip("torch")
    from paper_0812_0244_gb300.autograd import vdw_energy
    gen = torch.Generator().manual_seed(3)
    n = torch.rand(4, 5, 6, generator=gen, requires_grad=wants != "grad")
    grad = torch.rand(3, 4, 5, 6, generator=gen, requires_grad=wants != "n")
    E = vdw_energy(n, grad, Stub())
    ins = [t for t in (n, grad) if t.requires_grad]
    scales = torch.tensor([1.0, -2.0, 0.5], dtype=torch.float64)
    if route == "batched":
        got = torch.autograd.grad(E, ins, grad_outputs=scales, is_grads_batched=True)
    else:
        got = [torch.stack(p) for p in zip(*(
            torch.autograd.grad(E, ins, grad_outputs=s, retain_graph=True, create_graph=route == "create_graph")
            for s in scales))]
    for t, g in zip(ins, got):
        want = 2 * t if t is n else 3 * t ** 2
        for k in range(3):
            # a few FP32 roundings of products
            torch.testing.assert_close(g[k], want * float(scales[k]), rtol=1e-6, atol=0)
