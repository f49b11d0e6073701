"""Calls captured into a CUDA graph and replayed on new inputs give the eager
results to the bit: the launches that may overlap their predecessors and the
side stream of the energy reduction keep their order under capture, and the
count of invalid points is that of the call that ran last."""
import numpy as np
import pytest

from paper_0812_0244_gb300 import synthetic as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(12, 15, 16), (24, 24, 24), (72, 90, 90)])
@pytest.mark.parametrize("kind", ["ev", "energy", "w", "xc", "fd"])
def test_replay_equals_eager(shape, kind):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0812_0244_gb300 import vdwnl
    ctx = vdwnl.VdwNL(vdwnl.Params(Nq=8, na=48, Nr=512, Nk=512))
    d = [S.two_atom_density(k, shape=shape) for k in range(2)]
    ctx.plan(shape, d[0]["L"])
    ins = [(torch.tensor(x["n"].astype(np.float32), device="cuda"),
            torch.tensor(x["grad"].astype(np.float32), device="cuda")) for x in d]
    ins[1][0].reshape(-1)[3:20] = -1.0
    n, g = (t.clone() for t in ins[0])
    E = torch.zeros(4, dtype=torch.float64, device="cuda")
    v, w = torch.zeros_like(n), torch.zeros_like(g)

    def call():
        if kind == "ev":
            ctx.energy_potential(n, g, E, v)
        elif kind == "energy":
            ctx.energy_potential(n, g, E)
        elif kind == "w":
            ctx.energy_potential(n, g, None, v, w)
        elif kind == "xc":
            E.copy_(ctx.xc_energy_potential(n, v=v)[0])
        else:
            ctx.energy_potential_fd(n, E=E, v=v)

    call()  # the buffers of the library's own gradient
    torch.cuda.synchronize()
    eager = []
    for k in range(2):
        n.copy_(ins[k][0]), g.copy_(ins[k][1])
        call()
        eager.append([t.clone() for t in (E, v, w)] + [ctx.invalid_points()])
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call()
    for k in (1, 0, 1):
        n.copy_(ins[k][0]), g.copy_(ins[k][1])
        for t in (E, v, w):
            t.zero_()
        if kind == "energy":
            v.copy_(eager[k][1])
        if kind != "w":
            w.copy_(eager[k][2])
        graph.replay()
        torch.cuda.synchronize()
        for a, b in zip((v, w), eager[k][1:3]):
            assert torch.equal(a, b)
        if kind != "w":
            assert torch.equal(E, eager[k][0])
        assert ctx.invalid_points() == eager[k][3] == (17 if k else 0)
