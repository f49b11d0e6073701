"""Launches of thousands of small planes, more than 32 per SM: long y axes of
one density against the FP64 oracle, and batches against single calls.

Tolerances of the parity tests: E to 1e-6 Ha, v to 1e-5 of max|v|; a batch
gives the single calls' results to the bit."""
import numpy as np
import pytest

import oracle as O
from paper_0812_0244_gb300 import synthetic as S

pytestmark = pytest.mark.gpu

KW = dict(Nq=20, q_1=0.1, lam=1.2, na=48, Nr=512, Nk=512)


@pytest.fixture(scope="module")
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0812_0244_gb300 import vdwnl
    return vdwnl.VdwNL(vdwnl.Params(**KW))


@pytest.mark.parametrize("shape", [(24, 250, 24), (32, 256, 32), (16, 256, 16)])
def test_long_y_axis(ctx, shape):
    import torch
    L = 0.45 * np.array(shape[::-1], np.float64)
    z, y, x = np.meshgrid(*[2 * np.pi * np.arange(s) / s for s in shape], indexing="ij")
    # 0.2 Ha at most: the FP32 pointwise chain's share of E stays below the tolerance
    n = (0.004 * (1 + 0.3 * np.cos(x) * np.cos(y) + 0.3 * np.sin(z + 0.4))).astype(np.float32)
    g = O.spectral_gradient(n.astype(np.float64), L).astype(np.float32)
    ref = O.energy_potential(n.astype(np.float64), g.astype(np.float64), L, O.kernel_table(O.Params(**KW)))
    ctx.plan(shape, L)
    E, v, _ = ctx.compute(torch.tensor(n, device="cuda"), torch.tensor(g, device="cuda"))
    E, v = E.cpu().numpy(), v.cpu().numpy()
    assert abs(E[0] - ref["E"]) <= 1e-6, (E, ref["E"])
    assert np.abs(v - ref["v"]).max() <= 1e-5 * np.abs(ref["v"]).max()


@pytest.mark.parametrize("n,B", [(24, 16), (24, 11), (32, 8), (30, 10)])
def test_batches_of_small_cubes(ctx, n, B):
    import torch
    shape = (n, n, n)
    ds = [S.two_atom_density(b, shape=shape) for b in range(B)]
    ctx.plan(shape, ds[0]["L"])
    nt = torch.tensor(np.stack([d["n"] for d in ds]).astype(np.float32), device="cuda")
    gt = torch.tensor(np.stack([d["grad"] for d in ds]).astype(np.float32), device="cuda")
    ctx.plan_batch(B)
    E, v = ctx.energy_potential_batched(nt, gt, v=torch.empty_like(nt))
    for b in range(B):
        E1, v1, _ = ctx.compute(nt[b].contiguous(), gt[b].contiguous())
        assert torch.equal(E[b], E1) and torch.equal(v[b], v1), b
