"""The work that users of this framework have it do, as timed cases.

listed() and draw(rng) give cases (dicts of plain values), prepare(case, seed)
the density and the planned context that a program holds before its call,
run(state) one pass through the public entry points, work(case) the bytes and
operations such a pass cannot do without, and exact(case, seed) the pass's
outputs in 64-bit arithmetic, stated here in plain torch.

Fields of a case: "kind" (the entry point), n1, n2, n3 (grid), Nq (mesh of the
interpolation), B (densities per call), "cell" (what is in it: "atoms" and
"tube" have vacuum at a density floor of 1e-6, "solid" fills its cell), h (grid
spacing, bohr).
"""
import math

import numpy as np
import torch

from paper_0812_0244_gb300 import learned as LR
from paper_0812_0244_gb300 import vdwnl
from paper_0812_0244_gb300.autograd import vdw_energy

BOHR_PER_ANG = 1.0 / 0.529177210903
# The kernel table of the test suite's lighter quadrature with the default
# radial mesh: the table is made once per program and enters the timed work
# only through Nq and Nk.
TABLE = dict(na=128, Nr=2048)


# --------------------------------------------------------------------------
# cases
# --------------------------------------------------------------------------

def _case(name, kind, n1, n2, n3, h, cell="atoms", Nq=20, B=1):
    return dict(name=name, kind=kind, n1=n1, n2=n2, n3=n3, h=h, cell=cell, Nq=Nq, B=B)


def listed():
    return [
        # a dimer in a 10 A box at 24^3: the smallest grid in daily use, one
        # SCF step of a small molecule; launches and latency count
        _case("dimer_24_ev", "ev", 24, 24, 24, 0.787),
        # the same box at its production grid, inside a torch program that
        # differentiates the energy (forward and backward)
        _case("dimer_48_autograd", "autograd", 48, 48, 48, 0.394),
        # a molecule in an oblong box, ragged sizes with an odd N2, 12 mesh
        # points: the energy alone (line searches, post-SCF evaluation)
        _case("molecule_60x75x54_energy", "energy", 60, 75, 54, 0.36, Nq=12),
        # a crystal cell: the whole E_xc and v_xc of an SCF step, the library
        # making the spectral gradient itself
        _case("solid_100_xc", "xc", 100, 100, 100, 0.30, cell="solid"),
        # a larger crystal cell with the paper's finite-difference gradient
        _case("solid_128_fd", "fd", 128, 128, 128, 0.28, cell="solid"),
        # the wall scan and the training targets: eight rigid translations or
        # samples of a tube per call, on the scan's coarse and fine grids
        _case("tube_144_batch8", "batch", 144, 144, 72, 0.328, cell="tube", B=8),
        _case("tube_200_batch4", "batch", 200, 200, 72, 0.236, cell="tube", B=4),
        # one SCF step of the double-wall tube, the benchmark's workload, on
        # device buffers and from a host program's buffers
        _case("tube_180_ev", "ev", 180, 180, 72, 0.2625, cell="tube"),
        _case("tube_180_host", "host", 180, 180, 72, 0.2625, cell="tube"),
        # the paper's own mesh cutoff for that tube, differentiated in torch
        _case("tube_256_autograd", "autograd", 256, 256, 96, 0.1845, cell="tube"),
        # the learned 8-channel basis: inference from its tabulated network,
        # and a training step (parameter gradients, update, reload)
        _case("tube_180_learned", "learned", 180, 180, 72, 0.2625, cell="tube"),
        _case("tube_180_train", "train", 180, 180, 72, 0.2625, cell="tube"),
    ]


def _smooth(lo, hi, even):
    out = []
    for n in range(lo, hi + 1):
        m = n
        for p in (2, 3, 5):
            while m % p == 0:
                m //= p
        if m == 1 and not (even and n % 2):
            out.append(n)
    return out


def _log_pick(rng, sizes):
    """One of sizes, evenly over their logarithm."""
    x = math.exp(rng.uniform(math.log(sizes[0]), math.log(sizes[-1])))
    return min(sizes, key=lambda n: abs(math.log(n / x)))


def draw(rng):
    kind = rng.choice(["ev", "ev", "energy", "autograd", "xc", "fd", "batch", "host", "learned"])
    while True:
        n1 = _log_pick(rng, _smooth(20, 256, True))
        n2 = _log_pick(rng, _smooth(20, 256, False))
        n3 = _log_pick(rng, _smooth(20, 200, True))
        B = rng.randint(2, 8) if kind == "batch" else 1
        if (n1 // 2 + 1) * n3 <= 20000 and n1 * n2 * n3 * B <= 6300000:
            break
    cell = "solid" if kind in ("xc", "fd") else rng.choice(["atoms", "solid"])
    Nq = 20 if kind == "learned" else rng.choice([20, 20, 20, 16, 12, 8])
    c = _case("", kind, n1, n2, n3, round(rng.uniform(0.265, 0.42), 4), cell=cell, Nq=Nq, B=B)
    del c["name"]
    return c


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------

def _device():
    return torch.device("cuda", torch.cuda.current_device())


def _edges(case):
    if case["cell"] == "tube":  # four axial periods of an armchair tube in a 25 A square cell
        return np.array([25.0, 25.0, 9.84]) * BOHR_PER_ANG
    return np.array([case["n1"], case["n2"], case["n3"]]) * case["h"]


def _sites(case, rng, L):
    if case["cell"] == "tube":  # (5,5)@(10,10): four atoms per repeat, rings of 5 and 10 repeats
        out = []
        for rep, shift, rot in ((5, 0.0, 0.0), (10, rng.uniform(0, 2.46), rng.uniform(0, 0.6))):
            R = 3.0 * 1.42 * rep / (2 * math.pi)
            for k in range(4):
                for j in range(rep):
                    for s, z in ((0.0, 0.0), (1.42, 0.0), (2.13, 1.23), (3.55, 1.23)):
                        phi = (j * 4.26 + s) / R + rot
                        out.append((R * math.cos(phi) + 12.5, R * math.sin(phi) + 12.5, k * 2.46 + z + shift))
        return np.array(out) * BOHR_PER_ANG
    if case["cell"] == "solid":  # a jittered simple lattice, about 5 bohr apart
        m = [max(1, int(round(x / 5.0))) for x in L]
        g = np.stack(np.meshgrid(*[np.arange(k) / k for k in m], indexing="ij"), -1).reshape(-1, 3)
        return (g + rng.uniform(-0.03, 0.03, g.shape) / np.array(m)) * L
    # a molecule of a few atoms about the middle of the box
    k = int(min(12, max(2, round(float(np.prod(L)) / 3000.0))))
    return 0.5 * L + rng.uniform(-0.22, 0.22, (k, 3)) * L


def _density(case, seed, k, device):
    """Density k of the case: a sum of two Gaussians per site, FP32, and its
    spectral gradient (evaluated in 64 bits, rounded to FP32)."""
    rng = np.random.default_rng((int(seed), k))
    L = _edges(case)
    shape = (case["n3"], case["n2"], case["n1"])
    sites = _sites(case, rng, L)
    w = rng.uniform(0.3, 0.7, len(sites))
    cen = np.concatenate([sites, sites])
    sig = rng.uniform(0.4, 1.2, len(cen)) + (0.5 if case["cell"] == "solid" else 0.0)
    if case["h"] > 0.5:  # what a coarse grid can carry
        sig = sig + 0.4
    amp = 4.0 * np.concatenate([w, 1 - w]) / ((2 * math.pi) ** 1.5 * sig ** 3)
    s = torch.tensor(sig, dtype=torch.float64, device=device)[:, None]
    prof = []
    for d, nd in ((0, case["n1"]), (1, case["n2"]), (2, case["n3"])):
        x = torch.arange(nd, dtype=torch.float64, device=device) * (L[d] / nd)
        dx = x[None] - torch.tensor(cen[:, d], device=device)[:, None]
        dx = dx - L[d] * torch.round(dx / L[d])
        prof.append(sum(torch.exp(-(dx + i * L[d]) ** 2 / (2 * s * s)) for i in (-1, 0, 1)))
    px, py, pz = prof
    yx = (py[:, :, None] * px[:, None, :]).reshape(len(cen), -1)
    n = ((pz * torch.tensor(amp, device=device)[:, None]).T @ yx).reshape(shape) + 1e-6
    n = n.to(torch.float32)
    return n, _derivative(n.double(), L).to(torch.float32)


def _wave(shape, L, device, keep_nyquist):
    """Components of G on the half spectrum (x last, non-negative frequencies)."""
    out = []
    for ax, (nd, l) in enumerate(zip(shape, L[::-1])):
        m = torch.fft.rfftfreq(nd, 1.0 / nd, dtype=torch.float64, device=device) if ax == 2 else \
            torch.fft.fftfreq(nd, 1.0 / nd, dtype=torch.float64, device=device)
        if nd % 2 == 0 and not keep_nyquist:
            m = torch.where(m.abs() * 2 == nd, torch.zeros_like(m), m)
        out.append((2 * math.pi / l * m).reshape([-1 if i == ax else 1 for i in range(3)]))
    return out[::-1]  # x, y, z


def _derivative(f, L):
    fh = torch.fft.rfftn(f)
    return torch.stack([torch.fft.irfftn(1j * g * fh, s=f.shape) for g in _wave(f.shape, L, f.device, False)])


def _stencil(f, L):
    return torch.stack([(torch.roll(f, -1, 2 - d) - torch.roll(f, 1, 2 - d)) * (f.shape[2 - d] / (2 * L[d]))
                        for d in range(3)])


_kept = {}  # the program's kernel tables by Nq, and its one planned context


def _params(Nq):
    return vdwnl.Params(Nq=Nq, **TABLE)


def _context(case):
    key = (case["kind"], case["n1"], case["n2"], case["n3"], case["Nq"], case["B"], case["h"], case["cell"])
    if _kept.get("key") != key:
        _kept.pop("ctx", None)
        if ("table", case["Nq"]) not in _kept:
            _kept["table", case["Nq"]] = vdwnl.kernel_table(_params(case["Nq"]))
        t = _kept["table", case["Nq"]]
        ctx = vdwnl.VdwNL(_params(case["Nq"]), phi_k=t["phi_k"], C_s=t["C_s"])
        ctx.plan((case["n3"], case["n2"], case["n1"]), _edges(case))
        if case["B"] > 1:
            ctx.plan_batch(case["B"])
        if case["kind"] == "learned":
            mdl = LR.load()
            ctx.learned_load(torch.tensor(mdl["params"], dtype=torch.float32, device=_device()), mdl["J"],
                             mdl["k_max"], mdl["feat"], mdl["base"])
            ctx.learned_tabulate(LR.TAB_T, LR.TAB_D)
        _kept["ctx"], _kept["key"] = ctx, key
    return _kept["ctx"]


def prepare(case, seed):
    dev = _device()
    kind = case["kind"]
    st = dict(kind=kind, ctx=_context(case))
    dens = [_density(case, seed, k, dev) for k in range(case["B"])]
    if kind == "batch":
        st["n"] = torch.stack([d[0] for d in dens]).contiguous()
        st["g"] = torch.stack([d[1] for d in dens]).contiguous()
        return st
    st["n"], st["g"] = dens[0][0].contiguous(), dens[0][1].contiguous()
    if kind == "host":
        st["n"] = st["n"].cpu().pin_memory().numpy()
        st["g"] = st["g"].cpu().pin_memory().numpy()
        st["v"] = torch.empty(st["n"].shape, dtype=torch.float32).pin_memory().numpy()
    elif kind == "autograd":
        st["n"].requires_grad_()
        st["g"].requires_grad_()
    elif kind == "train":
        mdl = LR.load()
        st["p"] = torch.tensor(mdl["params"], dtype=torch.float32, device=dev)
        st["mdl"] = mdl
    return st


# --------------------------------------------------------------------------
# one pass
# --------------------------------------------------------------------------

def run(st):
    ctx, kind, n, g = st["ctx"], st["kind"], st["n"], st["g"]
    if kind == "ev":
        E, v, _ = ctx.compute(n, g)
        return {"E": E, "v": v}
    if kind == "energy":
        E, _, _ = ctx.compute(n, g, want_v=False)
        return {"E": E}
    if kind == "autograd":
        E = vdw_energy(n, g, ctx)
        dn, dg = torch.autograd.grad(E, (n, g))
        return {"E": E.detach(), "dn": dn, "dg": dg}
    if kind == "xc":
        E, v = ctx.xc_energy_potential(n, v=torch.empty_like(n))
        return {"E": E, "v": v}
    if kind == "fd":
        E, v = ctx.energy_potential_fd(n, v=torch.empty_like(n))
        return {"E": E, "v": v}
    if kind == "batch":
        E, v = ctx.energy_potential_batched(n, g, v=torch.empty_like(n))
        return {"E": E, "v": v}
    if kind == "host":
        E, v = ctx.energy_potential_host(n, g, v=st["v"])
        return {"E": E, "v": v}
    if kind == "learned":
        E, v, _ = ctx.learned_compute(n, g)
        return {"E": E, "v": v}
    # one training step on one density, from the stored parameters: load, the
    # energy's parameter gradients, the update of the network and the knots
    mdl = st["mdl"]
    p = st["p"].clone()
    ctx.learned_load(p, mdl["J"], mdl["k_max"], mdl["feat"], mdl["base"])
    grad = torch.zeros(p.numel(), dtype=torch.float64, device=p.device)
    E = torch.empty(3, dtype=torch.float64, device=p.device)
    ctx.learned_param_grad(n, g, grad, coef=1.0, E=E)
    m, v2 = torch.zeros_like(p), torch.zeros_like(p)
    vdwnl.adam_step(p, grad, m, v2, 1, 1e-5)
    return {"E": E, "p": p, "m": m, "v2": v2}


# --------------------------------------------------------------------------
# what a pass cannot do without
# --------------------------------------------------------------------------

def work(case):
    N = case["n1"] * case["n2"] * case["n3"]
    kind = case["kind"]
    Nq = 8 if kind in ("learned", "train") else case["Nq"]
    pairs = Nq * (Nq + 1) // 2
    fft = 2.5 * N * math.log2(N)  # one real transform
    half = N * (case["n1"] // 2 + 1) / case["n1"]
    contract = half * 2 * (3 * pairs + 4 * (pairs - Nq) + 4 * Nq)
    energy = Nq * fft + contract + 200 * N
    pot = Nq * fft + 8 * Nq * N + (0 if kind in ("fd", "autograd") else 4 * fft)
    # inputs n and grad n (xc and fd read n alone), outputs v (autograd: dE/dn, dE/d grad n)
    ins = {"xc": 4, "fd": 4}.get(kind, 16)
    outs = {"energy": 0, "autograd": 16, "train": 0}.get(kind, 4)
    flops = energy + (0 if kind == "energy" else pot)
    if kind == "xc":
        flops += 4 * fft + 150 * N
    if kind == "train":  # backward through a 2-64-64-8 network at every point
        flops += N * 6 * (2 * 64 + 64 * 64 + 64 * 8)
        ins += 0.0
    return {"bytes": float(case["B"] * N * (ins + outs)), "flops": float(case["B"] * flops)}


# --------------------------------------------------------------------------
# the outputs in 64 bits
# --------------------------------------------------------------------------

def _q_mesh(Nq, q1=1e-5, lam=1.2, qc=5.0):
    a = np.arange(Nq, dtype=np.float64)
    return q1 + (qc - q1) * (lam ** a - 1.0) / (lam ** (Nq - 1) - 1.0)


def _spline_M(x, Y):
    """Second derivatives at the knots of the natural cubic splines through the columns of Y."""
    n, h = len(x), np.diff(x)
    A, R = np.eye(n), np.zeros((n, Y.shape[1]))
    for i in range(1, n - 1):
        A[i, i - 1:i + 2] = h[i - 1], 2 * (h[i - 1] + h[i]), h[i]
        R[i] = 6 * ((Y[i + 1] - Y[i]) / h[i] - (Y[i] - Y[i - 1]) / h[i - 1])
    return np.linalg.solve(A, R)


def _dion(d1, d2, dev):
    """The kernel phi(d1, d2) of Dion et al. by double quadrature; differentiable in d1 and d2."""
    x, w = np.polynomial.legendre.leggauss(TABLE["na"])
    T = math.atan(64.0)
    a = torch.tensor(np.tan(0.5 * T * (x + 1)), device=dev)
    wa = torch.tensor(0.5 * T * w, device=dev) * (1 + a * a)
    s, c = torch.sin(a), torch.cos(a)
    j0 = s / a
    a2 = a * a  # (sin a - a cos a) / a^3, by its series where that cancels
    kf = torch.where(a < 0.3, 1 / 3 - a2 / 30 + a2 ** 2 / 840 - a2 ** 3 / 45360 + a2 ** 4 / 3991680, (s - a * c) / a ** 3)
    W = 2 * (j0[:, None] * kf + kf[:, None] * j0 - 3 * kf[:, None] * kf)
    K = (2 / math.pi ** 2) * (wa * a2)[:, None] * (wa * a2) * W
    out = []
    for b1, b2 in zip(d1.split(256), d2.split(256)):
        def nu(d):
            return a2 / (2 * -torch.expm1(-(4 * math.pi / 9) * a2 / d[:, None] ** 2))
        n1, n2 = nu(b1), nu(b2)
        wx, yz = n1[:, :, None] + n1[:, None], n2[:, :, None] + n2[:, None]
        wy = (n1 + n2)
        wz = n1[:, :, None] + n2[:, None]
        yx = n2[:, :, None] + n1[:, None]
        t = 0.5 * (1 / wx + 1 / yz) * (1 / (wy[:, :, None] * wy[:, None]) + 1 / (wz * yx))
        out.append((t * K).sum((1, 2)))
    return torch.cat(out)


def _phi(d1, d2, dev):
    """phi(d1, d2) with its closed-form limit where both arguments reach 8."""
    lim = -12 * (4 * math.pi / 9) ** 3 / (d1 ** 2 * d2 ** 2 * (d1 ** 2 + d2 ** 2))
    near = torch.minimum(d1, d2) < 8.0
    out = lim.clone()
    if near.any():
        out[near] = _dion(d1[near], d2[near], dev)
    return out


def _slope(c, s, dev):
    """phi and its derivative along the ray (c, s) d at d = 1."""
    with torch.enable_grad():
        t = torch.ones_like(c, requires_grad=True)
        f = _dion(c * t, s * t, dev)
        return f.detach(), torch.autograd.grad(f.sum(), t)[0]


def _kernel_table(Nq, dev):
    """(q mesh, radial table [pairs][Nk] of phi_ab(k) with its spline's second derivatives, C_s)."""
    if ("exact", Nq) in _kept:
        return _kept["exact", Nq]
    rc, kmax, Nk, Nr = 100.0, 40.0, 1024, TABLE["Nr"]
    r2 = torch.full((1,), math.sqrt(0.5), dtype=torch.float64, device=dev)
    f, df = _slope(r2, r2, dev)
    phi0 = f - 0.5 * df

    def soft(c, s):
        f, df = _slope(c, s, dev)
        p4 = phi0 - f + 0.5 * df
        return 0.5 * df - 2 * p4, p4

    x, w = np.polynomial.legendre.leggauss(64)
    X = math.sqrt(0.5)
    xs = torch.tensor(0.5 * X * (x + 1), device=dev)
    p2, p4 = soft(r2, r2)
    Cs = float((torch.tensor(0.5 * X * w, device=dev) * 4 * math.pi * xs ** 2
                * (_phi(xs, xs, dev) - (phi0 + p2 * 2 * xs ** 2 + p4 * 4 * xs ** 4))).sum())
    qm = _q_mesh(Nq)
    r = torch.linspace(0, rc, Nr + 1, dtype=torch.float64, device=dev)
    rows = []
    for a in range(Nq):
        for b in range(a, Nq):
            qq = math.hypot(qm[a], qm[b])
            d = qq * r
            p2, p4 = soft(torch.full_like(r2, qm[a] / qq), torch.full_like(r2, qm[b] / qq))
            y = phi0 + p2 * d ** 2 + p4 * d ** 4
            far = d >= 1.0
            if far.any():
                y[far] = _phi(qm[a] * r[far], qm[b] * r[far], dev)
            rows.append(y)
    simpson = torch.ones(Nr + 1, dtype=torch.float64, device=dev)
    simpson[1:-1:2], simpson[2:-1:2] = 4.0, 2.0
    k = torch.linspace(0, kmax, Nk, dtype=torch.float64, device=dev)
    J = torch.sinc(k[:, None] * r / math.pi) * (4 * math.pi * (rc / Nr / 3) * simpson * r * r)
    tab = torch.stack(rows) @ J.T
    M = torch.tensor(_spline_M(k.cpu().numpy(), tab.T.cpu().numpy()).T.copy(), device=dev)
    _kept["exact", Nq] = (qm, tab, M, kmax / (Nk - 1), Cs)
    return _kept["exact", Nq]


def _lda(rs):
    b = (7.5957, 3.5876, 1.6382, 0.49294)
    s = torch.sqrt(rs)
    return -0.062182 * (1 + 0.2137 * rs) * torch.log1p(1 / (0.062182 * (b[0] * s + b[1] * rs + b[2] * rs * s + b[3] * rs * rs)))


def _saturated_q(n, g2):
    kF = (3 * math.pi ** 2 * n) ** (1 / 3)
    rs = (3 / (4 * math.pi * n)) ** (1 / 3)
    q0 = kF * (1 + 0.8491 / 9 * g2 / (4 * kF ** 2 * n ** 2)) - 4 * math.pi / 3 * _lda(rs)
    y = torch.clamp(q0 / 5.0, max=50.0)
    return 5.0 * -torch.expm1(-sum(y ** m / m for m in range(1, 13)))


def _weights(q, qm):
    """The cardinal splines p_a(q), one after another."""
    M = torch.tensor(_spline_M(qm, np.eye(len(qm))).T.copy(), device=q.device)
    x = torch.tensor(qm, device=q.device)
    qc = torch.clamp(q, qm[0], qm[-1])
    k = torch.clamp(torch.searchsorted(x, qc.detach(), right=True) - 1, 0, len(qm) - 2)
    h = x[k + 1] - x[k]
    A = (x[k + 1] - qc) / h
    B = 1 - A
    c0, c1 = (A ** 3 - A) * h * h / 6, (B ** 3 - B) * h * h / 6
    for a in range(len(qm)):
        yield A * (k == a) + B * (k + 1 == a) + c0 * M[a][k] + c1 * M[a][k + 1]


def _network(n, g2, mdl):
    """The 8 outputs of the stored 2-64-64-8 network (activations not rounded)."""
    dev = n.device
    p = torch.tensor(mdl["params"], dtype=torch.float32, device=dev)
    W1, b1, W2, b2, W3, b3 = (x.reshape(s) for x, s in zip(
        torch.split(p[:LR.OFF_K], [128, 64, 4096, 64, 512, 8]), [(64, 2), (64,), (64, 64), (64,), (8, 64), (8,)]))
    r = [x.bfloat16().double() for x in (W1, W2, W3)]
    mu1, s1, mu2, s2, eps = mdl["feat"]
    x1 = torch.clamp((torch.log(n) - mu1) / s1, -LR.TAB_D, LR.TAB_D)
    x2 = torch.clamp((0.5 * torch.log(g2 * n ** (-8 / 3) + eps ** 2) - mu2) / s2, -LR.TAB_D, LR.TAB_D)
    h = torch.nn.functional.silu(torch.stack([x1, x2], -1) @ r[0].T + b1.double())
    h = torch.nn.functional.silu(h @ r[1].T + b2.double())
    return h @ r[2].T + b3.double()


def _channels(n, g2, case, qm, mdl):
    """theta_a = n w_a of every channel, and q."""
    q = _saturated_q(n, g2)
    if mdl is None:
        return [n * p for p in _weights(q, qm)], torch.clamp(q, qm[0], qm[-1])
    o = _network(n, g2, mdl)
    bm = _q_mesh(8, mdl["base"][0], mdl["base"][1])
    qp = _q_mesh(case["Nq"])
    return [n * (p + o[..., a]) for a, p in enumerate(_weights(q, bm))], torch.clamp(q, qp[0], qp[-1])


def _pair_kernels(case, G, mdl, dev):
    """phi_ab(|G|) of each pair a <= b, one after another."""
    if mdl is None:
        _, tab, M, dk, _ = _kernel_table(case["Nq"], dev)
        j = torch.clamp((G / dk).long(), 0, tab.shape[1] - 2)
        B = G / dk - j
        A = 1 - B
        c0, c1 = (A ** 3 - A) * dk * dk / 6, (B ** 3 - B) * dk * dk / 6
        for y, m in zip(tab, M):
            yield A * y[j] + B * y[j + 1] + c0 * m[j] + c1 * m[j + 1]
        return
    K = torch.tensor(mdl["params"][LR.OFF_K:], dtype=torch.float64, device=dev).reshape(36, mdl["J"])
    K = torch.cat([K[:, 1:2], K, 2 * K[:, -1:] - K[:, -2:-1]], 1)  # even in k; linear past the last knot
    dk = mdl["k_max"] / (mdl["J"] - 1)
    j = torch.clamp((G / dk).long(), 0, mdl["J"] - 2)
    t = G / dk - j
    w = [(-t ** 3 + 2 * t ** 2 - t) / 2, (3 * t ** 3 - 5 * t ** 2 + 2) / 2, (-3 * t ** 3 + 4 * t ** 2 + t) / 2, (t ** 3 - t ** 2) / 2]
    for y in K:
        yield sum(wi * y[j + i] for i, wi in enumerate(w))


def _functional(case, n32, g32, mdl):
    """E [3], v_loc, w [3] and the semilocal sums of one density."""
    dev = n32.device
    L = _edges(case)
    n = n32.double().requires_grad_()
    g = g32.double().requires_grad_()
    N, Omega = n.numel(), float(np.prod(L))
    qm, _, _, _, Cs = _kernel_table(case["Nq"], dev)
    with torch.no_grad():
        th = torch.stack([torch.fft.rfftn(t) for t in _channels(n, (g * g).sum(0), case, qm, mdl)[0]])
        G = torch.sqrt(sum(x * x for x in _wave(n.shape, L, dev, True)))
        u = torch.zeros_like(th)
        pairs = _pair_kernels(case, G, mdl, dev)
        for a in range(len(th)):
            for b in range(a, len(th)):
                f = next(pairs)
                u[a] += f * th[b]
                if b != a:
                    u[b] += f * th[a]
        wt = torch.full((n.shape[2] // 2 + 1,), 2.0, dtype=torch.float64, device=dev)
        wt[0] = wt[-1] = 1.0
        soft = 0.5 * Omega / N ** 2 * float((wt * (th.real * u.real + th.imag * u.imag).sum(0)).sum())
        del th
        ur = torch.stack([torch.fft.irfftn(x, s=n.shape) for x in u])
        del u, G
    sl = None
    with torch.enable_grad():
        theta, q = _channels(n, (g * g).sum(0), case, qm, mdl)
        dE = Cs * n ** 2 / (2 * q ** 3)
        S = sum((x * t).sum() for x, t in zip(ur, theta)) + dE.sum()
        if case["kind"] == "xc":
            kF = (3 * math.pi ** 2 * n) ** (1 / 3)
            s2 = (g * g).sum(0) / (4 * kF ** 2 * n ** 2)
            mu = 0.066725 * math.pi ** 2 / 3
            ex = -0.75 * (3 / math.pi) ** (1 / 3) * n ** (4 / 3) * (2.245 - 1.245 / (1 + mu * s2 / 1.245))
            ec = n * _lda((3 / (4 * math.pi * n)) ** (1 / 3))
            S = S + ex.sum() + ec.sum()
            sl = (float(ex.sum()) * Omega / N, float(ec.sum()) * Omega / N)
        vl, w = torch.autograd.grad(S, (n, g))
    corr = float(dE.sum()) * Omega / N
    return torch.tensor([soft + corr, soft, corr], dtype=torch.float64, device=dev), vl, w, sl


def exact(case, seed):
    dev, kind = _device(), case["kind"]
    L = _edges(case)
    dO = float(np.prod(L)) / (case["n1"] * case["n2"] * case["n3"])
    mdl = LR.load() if kind in ("learned", "train") else None
    Es, vs = [], []
    for k in range(case["B"]):
        n, g = _density(case, seed, k, dev)
        if kind == "xc":
            g = _derivative(n.double(), L)
        elif kind == "fd":
            g = _stencil(n.double(), L)
        E, vl, w, sl = _functional(case, n, g, mdl)
        if kind == "energy":
            return {"E": E}
        if kind == "train":  # the update rests on gradients through bf16 roundings: no 64-bit value
            return {"E": E, "p": None, "m": None, "v2": None}
        if kind == "autograd":
            return {"E": E[0], "dn": vl * dO, "dg": w * dO}
        D = _stencil if kind == "fd" else _derivative
        v = vl - sum(D(w[c].detach(), L)[c] for c in range(3))
        if sl is not None:
            E = torch.tensor([E[0] + sum(sl), E[0], sl[0], sl[1]], dtype=torch.float64, device=dev)
        Es.append(E)
        vs.append(v)
    if kind == "batch":
        return {"E": torch.stack(Es), "v": torch.stack(vs)}
    return {"E": Es[0], "v": vs[0]}
