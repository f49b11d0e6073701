"""Every line length the transforms take, in each direction, against the FP64
oracle: energy and potential on thin grids with the length along x, y or z,
and the spectral gradient.  The lengths cover every pair of radix groups, the
padded and ragged pencil tiles and the smallest and largest lines.

Tolerances: those of the parity tests for E (1e-6 Ha) and v (1e-5 of max|v|).
The spectral gradient's transforms round each coefficient by a few FP32 ulp of
the field's norm (six line transforms of at most five radices, 6e-8 each, all
adding up: below 2e-6), which the derivative scales by at most |G|max: the
error's norm is below 2e-6 |G|max times the field's.
"""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

LENGTHS = [n for n in range(4, 257) if 2 ** 8 * 3 ** 5 * 5 ** 3 % n == 0]
KW = dict(Nq=8, q_1=0.1, lam=1.45, na=48, Nr=512, Nk=512)


@pytest.fixture(scope="module")
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0812_0244_gb300 import vdwnl
    return vdwnl.VdwNL(vdwnl.Params(**KW))


@pytest.fixture(scope="module")
def tab():
    return O.kernel_table(O.Params(**KW))


def check(ctx, tab, shape, energy=True):
    import torch
    L = 0.45 * np.array(shape[::-1], np.float64)
    rng = np.random.default_rng(sum(shape))
    z, y, x = np.meshgrid(*[2 * np.pi * np.arange(s) / s for s in shape], indexing="ij")
    n = 0.05 * (1 + 0.3 * np.cos(x) * np.cos(y) + 0.3 * np.sin(z + 0.4)) * (1 + 0.02 * rng.uniform(-1, 1, shape))
    n = n.astype(np.float32)
    g = O.spectral_gradient(n.astype(np.float64), L)
    ctx.plan(shape, L)
    nt = torch.tensor(n, device="cuda")
    d = ctx.spectral_gradient(nt).cpu().numpy().astype(np.float64) - g
    gmax = np.pi / 0.45 * np.sqrt(3.0)
    assert np.linalg.norm(d) <= 2e-6 * gmax * np.linalg.norm(n), (shape, np.linalg.norm(d))
    g = g.astype(np.float32)
    ref = O.energy_potential(n.astype(np.float64), g.astype(np.float64), L, tab)
    E, v, _ = ctx.compute(nt, torch.tensor(g, device="cuda"))
    E, v = E.cpu().numpy(), v.cpu().numpy()
    if energy:
        assert abs(E[0] - ref["E"]) <= 1e-6 and abs(E[1] - ref["E_soft"]) <= 1e-6, (shape, E, ref["E"], ref["E_soft"])
    assert np.abs(v - ref["v"]).max() <= 1e-5 * np.abs(ref["v"]).max(), shape


@pytest.mark.parametrize("n", LENGTHS)
def test_line_length(ctx, tab, n):
    check(ctx, tab, (4, n, 6))
    if n % 2 == 0:
        check(ctx, tab, (6, 5, n))
        check(ctx, tab, (n, 9, 10))


@pytest.mark.parametrize("shape", [(200, 4, 250), (250, 4, 200), (256, 5, 200), (216, 4, 240), (200, 5, 256)])
def test_widest_planes(ctx, tab, shape):
    """Planes at the limit of shared memory, where the padded rows do not
    always fit.  Gradient and potential: these cells hold several Ha, of which
    1e-6 Ha is the FP32 pointwise chain's own share."""
    check(ctx, tab, shape, energy=False)
