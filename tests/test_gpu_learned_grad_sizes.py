"""Parameter gradients of the learned basis against the oracle at the sizes
where the 128-point tiles and the |G|-ordered runs go wrong: less than a tile,
a whole one, one and a remainder, several per team, points without density.

Tolerance: 2e-3 of each block's norm, as for the larger cells: an activation
that rounds to bf16 the other way (one in 3e-5) moves its own unit's share at
one point by 2^-9, which is below 2^-9 / sqrt(64) of a block's norm at 64 points.
"""
import numpy as np
import pytest

import oracle.learned as LO

pytestmark = pytest.mark.gpu

J, KMAX = 64, 30.0


@pytest.mark.parametrize("shape", [(4, 4, 4), (4, 8, 4), (4, 9, 4), (6, 25, 10), (40, 25, 40)])
def test_gradients(table, shape):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0812_0244_gb300 import vdwnl
    rng = np.random.default_rng(sum(shape))
    L = 0.5 * np.array(shape[::-1], np.float64)
    z, y, x = np.meshgrid(*[2 * np.pi * np.arange(s) / s for s in shape], indexing="ij")
    n = (0.05 * np.exp(0.8 * np.cos(x) * np.cos(y) + 0.5 * np.sin(z + 0.4))).astype(np.float32)
    g = (rng.normal(size=(3,) + shape) * 0.05).astype(np.float32)
    n.reshape(-1)[5::37] = 0.0
    n64, g64 = n.astype(np.float64), g.astype(np.float64)
    mdl = LO.random_model(41, J=J, k_max=KMAX, kscale=1e-3, mu=(-3.0, 0.0), sig=(1.0, 1.0), base=(0.6, 1.45))
    ctx = vdwnl.VdwNL(vdwnl.Params()).plan(shape, L)
    ctx.learned_load(torch.tensor(mdl.flat().astype(np.float32), device="cuda"), J, KMAX,
                     (mdl.mu1, mdl.sig1, mdl.mu2, mdl.sig2, mdl.eps), (mdl.base_q1, mdl.base_lam))
    nt, gt = torch.tensor(n, device="cuda"), torch.tensor(g, device="cuda")
    sizes = [int(np.prod(s)) for s in LO.LearnedModel.sizes(mdl.M, mdl.J)]
    offs = np.concatenate([[0], np.cumsum(sizes)])

    def compare(a, b, names):
        for k, name in enumerate(names):
            p, q = a[offs[k]:offs[k + 1]], b[offs[k]:offs[k + 1]]
            assert np.linalg.norm(p - q) <= 2e-3 * np.linalg.norm(q) + 1e-12, (name, np.linalg.norm(q))

    names = ["W1", "b1", "W2", "b2", "W3", "b3", "K"]
    gp = torch.zeros(offs[-1], dtype=torch.float64, device="cuda")
    ctx.learned_param_grad(nt, gt, gp, coef=1.0)
    compare(gp.cpu().numpy(), LO.energy_grad(n64, g64, L, mdl, table), names)
    target = rng.normal(0, 0.3, (8,) + shape).astype(np.float32)
    weight = (n / n.sum()).astype(np.float32)
    gp.zero_()
    ctx.learned_fit_grad(nt, gt, torch.tensor(target, device="cuda"), torch.tensor(weight, device="cuda"), gp)
    compare(gp.cpu().numpy(), LO.fit_grad(n64, g64, mdl, target.astype(np.float64), weight.astype(np.float64), 1e-12),
            names[:6])
    assert ctx.learned_status() == 0
