"""Timed cases of the VMC library: the calls a variational Monte Carlo program makes.

Amplitudes, local energies and log-derivatives of given configurations (measuring a
state), their autograd form, Markov-chain sampling of one and of several lattices, and
the stochastic-reconfiguration / tVMC step.  Lattices, bond dimensions and couplings are
those of the benchmark workloads and of the tests (Z2 with and without hard-core bosons,
Z3, Z4; D_k = 1..3).

Inputs.  Tensors are 1 + s N(0,1) on every symmetry-allowed block: the amplitudes of a
state near a ground state have a common sign or phase, unlike those of i.i.d. N(0,1)
tensors, whose sums cancel so far that single precision keeps few digits of E_loc on the
truncated lattices.  Starting configurations have plaquette powers uniform in Z_N and, with
matter, half filling.  The single-precision forms hand their numbers on in single
precision, which is what these hold; FP64 contexts in double.
"""

import math
import os
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import torch

import paper_2503_20566_gb300 as G
from paper_2503_20566_gb300.autograd import log_abs_psi

COUPLING = dict(h=1.0, g=0.33)
J_HOP = 0.5
CG = dict(diag_shift=1e-2, max_iter=20, tol=1e-10)


def _case(kind, name=None, N=2, Lx=8, Ly=8, D=4, chi=16, matter=False, cplx=False, precision="fp32", n=1):
    c = dict(kind=kind, N=N, Lx=Lx, Ly=Ly, D=D, chi=chi, matter=matter, cplx=cplx, precision=precision, n=n)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # the smallest call: a handful of amplitudes on the 3x3 boson lattice of the SR campaign
        _case("amplitude", "amplitude 3x3 bosons", Lx=3, Ly=3, D=6, chi=9, matter=True, n=16),
        # the largest lattice of the default benchmark: overlaps / reweighting on 32x32
        _case("amplitude", "amplitude 32x32 bosons", Lx=32, Ly=32, chi=24, matter=True, n=152),
        # measuring <E> of the 8x8 benchmark state, exact chi, many configurations
        _case("energy", "energy 8x8", n=2048),
        # ragged lattice, tensor-core (3-pass TF32) form, truncated
        _case("energy", "energy 12x9 bosons tf32", Lx=12, Ly=9, chi=16, matter=True, precision="tf32", n=304),
        # the Z3 workload: complex tensors, two powers of every plaquette
        _case("energy", "energy 16x16 Z3", N=3, Lx=16, Ly=16, D=6, chi=32, cplx=True, n=152),
        # gradients of the 16x16 lattice of the default benchmark
        _case("gradient", "gradient 16x16 bosons", Lx=16, Ly=16, chi=24, matter=True, n=304),
        # gradients of the tVMC workload: D_k = 3, complex
        _case("gradient", "gradient 10x10 D6", Lx=10, Ly=10, D=6, chi=36, cplx=True, n=152),
        # forward and backward through torch.autograd, odd sizes
        _case("autograd", "autograd 7x5 D6", Lx=7, Ly=5, D=6, chi=12, n=333),
        # one sampling call of short chains, exact chi, every output taken
        _case("sample", "sample 6x6", Lx=6, Ly=6, chi=8, n=256),
        # three lattices in one launch, truncated, reference precision
        _case("multi", "sample 9x7+7x7+5x6 bosons fp64", Lx=9, Ly=7, chi=6, matter=True, precision="fp64", n=96),
        # SR step of the 8x8 benchmark: more samples than parameters
        _case("sr", "sr 8x8", n=65536),
        # tVMC stage of the Z3 workload: fewer samples than parameters, complex
        _case("sr", "tvmc 16x16 Z3", N=3, Lx=16, Ly=16, D=6, chi=32, cplx=True, n=1024),
    ]


def _log_int(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    while True:
        kind = rng.choice(["amplitude", "energy", "gradient", "amplitude", "energy", "gradient", "autograd", "sample",
                           "multi", "sr"])
        N = rng.choice([2, 2, 2, 3, 4])
        Dk = rng.choice([1, 2, 2, 2, 3])
        Lx, Ly = _log_int(rng, 3, 24), _log_int(rng, 3, 24)
        chi = rng.randint(8, 36)
        cplx = N > 2 or rng.random() < 0.3
        matter = not cplx and rng.random() < 0.5
        precision = rng.choice(["fp32", "fp32", "fp32", "fp32", "tf32", "fp64"])
        n = _log_int(rng, 1, 2048)
        if kind == "autograd":
            cplx, N = False, 2
        if kind == "sample":
            # single precision at exact chi only: on a truncated lattice another rounding soon takes another Markov path
            precision = rng.choice(["fp32", "fp64"])
            if precision == "fp32":
                cplx, matter, N = False, False, 2
                Lx = min(Lx, 8 if Dk < 3 else 5)
                chi = max(chi, Dk ** (Lx // 2))
                n = min(n, 8000 // ((Lx - 1) * (Ly - 1)))
        if kind == "multi":
            precision, Lx, Ly = "fp64", max(5, min(Lx, 12)), max(5, min(Ly, 12))
        if kind == "sr":
            precision, n = rng.choice(["fp32", "fp32", "fp64"]), _log_int(rng, 256, 65536)
            Dk = max(Dk, 2)
        if precision == "tf32" and kind not in ("amplitude", "energy", "gradient"):
            precision = "fp32"
        if n < 1 or (Dk == 3 and min(Lx, Ly) < 4):
            continue
        c = _case(kind, N=N, Lx=Lx, Ly=Ly, D=Dk * N, chi=chi, matter=matter, cplx=cplx, precision=precision, n=n)
        # no costlier than the largest listed case (FP64 arithmetic runs at a small share of the FP32 rate)
        cost = work(c)["flops"] * (8 if precision == "fp64" else 1)
        if cost <= (2e10 if kind == "sr" else 1.5e10):
            return c


# ---- inputs -------------------------------------------------------------------
def _rng(seed, what):
    return np.random.default_rng([int(seed), what])


def _legs(c, x, y):
    return (x > 0, x < c["Lx"] - 1, y > 0, y < c["Ly"] - 1)


def _vertex_tables(c):
    """Blocks, entries per block and parameter offset of every vertex (row-major)."""
    Dk, nb, bs, off = c["D"] // c["N"], [], [], [0]
    for y in range(c["Ly"]):
        for x in range(c["Lx"]):
            k = sum(_legs(c, x, y))
            nb.append((2 if c["matter"] else 1) * c["N"] ** (k - 1))
            bs.append(Dk ** k)
            off.append(off[-1] + nb[-1] * bs[-1])
    return nb, bs, off


def _tensors(c, seed, n_params):
    r = _rng(seed, 1)
    if c["cplx"]:
        v = 1.0 + 0.85 * (r.standard_normal(n_params) + 1j * r.standard_normal(n_params))
        return v if c["precision"] == "fp64" else v.astype(np.complex64).astype(np.complex128)
    v = 1.0 + 0.5 * r.standard_normal(n_params)
    return v if c["precision"] == "fp64" else v.astype(np.float32).astype(np.float64)


def _configs(c, seed):
    """Physical starting configurations (n, [h][v][p]): links on a comb tree that
    satisfy the Gauss law for half filling, then random powers of every plaquette."""
    r, n, N, Lx, Ly = _rng(seed, 2), c["n"], c["N"], c["Lx"], c["Ly"]
    p = np.zeros((n, Ly * Lx), np.int64)
    if c["matter"]:
        bosons = Lx * Ly // 2 // N * N
        p[np.arange(n)[:, None], np.argsort(r.random((n, Lx * Ly)), axis=1)[:, :bosons]] = 1
    p = p.reshape(n, Ly, Lx)
    h, v = np.zeros((n, Ly, Lx - 1), np.int64), np.zeros((n, Ly - 1, Lx), np.int64)
    for x in range(Lx - 1, 0, -1):
        h[:, :, x - 1] = (h[:, :, x] if x < Lx - 1 else 0) - p[:, :, x]
    for y in range(Ly - 1):
        v[:, y, 0] = p[:, y, 0] + (v[:, y - 1, 0] if y else 0) - h[:, y, 0]
    t = r.integers(0, N, (n, Ly - 1, Lx - 1))
    h[:, :-1] += t
    v[:, :, 1:] += t
    h[:, 1:] -= t
    v[:, :, :-1] -= t
    return np.concatenate([a.reshape(n, -1) % N for a in (h, v)] + [p.reshape(n, -1)], axis=1).astype(np.int8)


def _samples(c, seed):
    """Samples as an SR step takes them: a block and its log-derivatives at every vertex.
    Samples near a node have large derivatives of all parameters, so scales differ."""
    r = _rng(seed, 3)
    nb, bs, _ = _vertex_tables(c)
    n, ns, D4 = c["n"], len(nb), (c["D"] // c["N"]) ** 4
    gen = torch.Generator(device="cuda").manual_seed(int(seed) * 7 + 5)
    bid = (torch.rand((n, ns), generator=gen, device="cuda") * torch.tensor(nb, device="cuda")).to(torch.int32)
    dt = torch.complex64 if c["cplx"] else torch.float32
    if c["precision"] == "fp64":
        dt = torch.complex128 if c["cplx"] else torch.float64
    scale = torch.exp(0.5 * torch.randn((n, 1, 1), generator=gen, device="cuda"))
    O = torch.empty((n, ns, D4), dtype=dt, device="cuda")
    for a in range(0, n, 4096):
        z = torch.randn((min(4096, n - a), ns, D4), generator=gen, device="cuda", dtype=dt)
        O[a:a + 4096] = (0.3 * z + 0.1) * scale[a:a + 4096]
    used = torch.arange(D4, device="cuda") < torch.tensor(bs, device="cuda")[:, None]
    O *= used
    e = torch.from_numpy(r.standard_normal(2 * n)).cuda()
    e[0::2] += O[:, 0, 0].real - 40.0
    if not c["cplx"]:
        e[1::2] = 0.0
    return dict(e_loc=e, block_ids=bid, O=O)


def _context(c, seed):
    ctx = G.Context(c["N"], c["Lx"], c["Ly"], c["D"], c["chi"], matter=c["matter"], J=J_HOP if c["matter"] else 0.0,
                    complex_=c["cplx"], precision=c["precision"], **COUPLING)
    ctx.set_tensors(_tensors(c, seed, ctx.n_params))
    return ctx


def _multi(c):
    """The lattices of a multi-context call: the case's and two smaller ones."""
    return [c, dict(c, Lx=c["Lx"] - 2), dict(c, Lx=max(3, c["Lx"] - 4), Ly=c["Ly"] - 1, n=c["n"] // 2 + 1)]


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "multi":
        cs = _multi(c)
        ctxs = [_context(q, seed + i) for i, q in enumerate(cs)]
        return dict(case=c, ctx=ctxs, seed=int(seed), cfg=[torch.from_numpy(_configs(q, seed + i)).cuda()
                                                           for i, q in enumerate(cs)])
    ctx = _context(c, seed)
    if kind == "sr":
        return dict(case=c, ctx=ctx, samples=_samples(c, seed))
    s = dict(case=c, ctx=ctx, seed=int(seed), cfg=torch.from_numpy(_configs(c, seed)).cuda())
    if kind == "autograd":
        dt = torch.float64 if c["precision"] == "fp64" else torch.float32
        s["theta"] = torch.from_numpy(_tensors(c, seed, ctx.n_params)).to("cuda", dt)
        s["weights"] = torch.from_numpy(_rng(seed, 4).standard_normal(c["n"])).cuda()
    return s


# ---- the passes -----------------------------------------------------------------
def _given(c, out):
    """The outputs in the precision that they hold."""
    if c["precision"] == "fp64":
        return out
    single = {torch.float64: torch.float32, torch.complex128: torch.complex64}
    return {k: v.to(single.get(v.dtype, v.dtype)) for k, v in out.items()}


def run(state):
    c, ctx = state["case"], state["ctx"]
    kind = c["kind"]
    if kind == "amplitude":
        la, ph = ctx.amplitude(state["cfg"])
        return _given(c, dict(log_abs=la, phase=ph))
    if kind == "energy":
        return _given(c, dict(e_loc=ctx.local_energy(state["cfg"])))
    if kind == "gradient":
        bid, O = ctx.log_grad(state["cfg"])
        return dict(block_ids=bid, O=O)
    if kind == "autograd":
        theta = state["theta"].detach().requires_grad_()
        la = log_abs_psi(theta, ctx, state["cfg"])
        (state["weights"] * la).sum().backward()
        return _given(c, dict(log_abs=la.detach(), grad=theta.grad))
    if kind == "sample":
        state["seed"] += 1
        out = ctx.sample_batch(state["cfg"], 1, state["seed"])
        return dict(_given(c, out), configs=state["cfg"])
    if kind == "multi":
        state["seed"] += 1
        outs = G.sample_multi(ctx, state["cfg"], 1, [state["seed"] + i for i in range(len(ctx))])
        return [dict(_given(c, o), configs=f) for o, f in zip(outs, state["cfg"])]
    mode = dict(mode=G.TDVP_STAGE1, dt=0.01) if c["cplx"] else dict(lr=0.01)
    st = ctx.sr_step(state["samples"], c["n"], **mode, **CG)
    stats, new = np.array([st[0], st[2], st[5]]), ctx.get_tensors()
    if c["precision"] == "fp64":
        return dict(stats=stats, tensors=new)
    return dict(stats=stats.astype(np.float32), tensors=new.astype(np.complex64 if c["cplx"] else np.float32))


# ---- what a pass cannot do without ----------------------------------------------
def work(case):
    c = case
    if c["kind"] == "multi":
        w = [work(dict(q, kind="sample")) for q in _multi(c)]
        return dict(bytes=sum(q["bytes"] for q in w), flops=sum(q["flops"] for q in w))
    nb, bs, off = _vertex_tables(c)
    n, ns, Dk = c["n"], len(nb), c["D"] // c["N"]
    sc = (16 if c["cplx"] else 8) if c["precision"] == "fp64" else (8 if c["cplx"] else 4)
    grad = n * (4.0 * ns + sc * sum(bs))
    if c["kind"] == "sr":
        # O is read once; every CG iteration forms O.p and O^H t of every sample
        return dict(bytes=grad + 16.0 * n + 2.0 * sc * off[-1],
                    flops=CG["max_iter"] * n * sum(bs) * 4.0 * (4 if c["cplx"] else 1))
    chi = min(c["chi"], Dk ** (min(c["Lx"], 40) // 2))
    # boundary absorption, per site: the leading costs of a single-layer contraction at cutoff chi
    site = 2.0 * (Dk ** 5 * chi ** 2 + Dk ** 4 * chi ** 2 + Dk ** 3 * chi ** 3) * (4 if c["cplx"] else 1)
    passes = dict(amplitude=1, energy=4, gradient=3, autograd=4, sample=8 if c["matter"] else 5)[c["kind"]]
    cfg = n * (2.0 * ns + c["Lx"] * (c["Ly"] - 1) + c["Ly"] * (c["Lx"] - 1)) / 2
    out = dict(amplitude=16.0 * n, energy=16.0 * n, gradient=grad, autograd=16.0 * n + 2 * sc * off[-1],
               sample=grad + 40.0 * n + cfg)[c["kind"]]
    return dict(bytes=cfg + sc * off[-1] + out, flops=n * ns * site * passes)


# ---- the same in 64 bits ----------------------------------------------------------
class _Net:
    """Configurations, blocks and boundary states of a case in plain numpy / torch FP64."""

    def __init__(self, c, seed):
        self.c, self.Dk, self.N = c, c["D"] // c["N"], c["N"]
        self.nb, self.bs, self.off = _vertex_tables(c)
        self.theta = torch.from_numpy(_tensors(c, seed, self.off[-1])).cuda()
        cfg = _configs(c, seed).astype(np.int64)
        Lx, Ly, n = c["Lx"], c["Ly"], c["n"]
        nh, nv = Ly * (Lx - 1), (Ly - 1) * Lx
        self.h = torch.from_numpy(cfg[:, :nh].reshape(n, Ly, Lx - 1)).cuda()
        self.v = torch.from_numpy(cfg[:, nh:nh + nv].reshape(n, Ly - 1, Lx)).cuda()
        self.p = torch.from_numpy(cfg[:, nh + nv:].reshape(n, Ly, Lx)).cuda()

    def block(self, x, y):
        """Index of the block that the configurations select at (x, y)."""
        legs = _legs(self.c, x, y)
        ch = [self.h[:, y, x - 1] if legs[0] else None, self.h[:, y, x] if legs[1] else None,
              self.v[:, y - 1, x] if legs[2] else None, self.v[:, y, x] if legs[3] else None]
        b = self.p[:, y, x].clone()
        for q in [q for q in ch if q is not None][:-1]:
            b = b * self.N + q
        return b

    def dims(self, x, y):
        return tuple(self.Dk if has else 1 for has in _legs(self.c, x, y))

    def tensor(self, x, y):
        v = y * self.c["Lx"] + x
        t = self.theta[self.off[v]:self.off[v + 1]].reshape((self.nb[v],) + self.dims(x, y))
        return t[self.block(x, y)]

    def row(self, y):
        return [self.tensor(x, y) for x in range(self.c["Lx"])]

    def boundary(self, rows, flip):
        """Boundary states after 0, 1, .. len(rows) rows (sites (n, left, physical, right)),
        with the log of their scale; `rows` in the order of absorption."""
        chi, host = self.c["chi"], [[t.cpu().numpy() for t in r] for r in rows]
        n = self.c["n"]

        def part(idx):
            dt = host[0][0].dtype
            M, lg, got = [np.ones((len(idx), 1, 1, 1), dt) for _ in host[0]], np.zeros(len(idx)), []
            got.append((M, lg))
            for r in host:
                new = []
                for A, W in zip(M, r):
                    W = W[idx].transpose(0, 1, 2, 4, 3) if flip else W[idx]  # [l][r][in][out]
                    Z = np.einsum("nadb,nlrdu->nalubr", A, W, optimize=True)
                    k, a, l, u, b, q = Z.shape
                    new.append(Z.reshape(k, a * l, u, b * q))
                R = np.ones((len(idx), 1, 1), dt)
                for i, Z in enumerate(new):
                    X = np.matmul(R, Z.reshape(len(idx), Z.shape[1], -1)).reshape(len(idx), -1, Z.shape[3])
                    u = Z.shape[2]
                    if i + 1 < len(new):
                        Q, R = np.linalg.qr(X)
                        f = np.linalg.norm(R, axis=(1, 2), keepdims=True)
                        R, lg = R / f, lg + np.log(f[:, 0, 0])
                        X = Q
                    new[i] = X.reshape(len(idx), -1, u, X.shape[2])
                C = np.ones((len(idx), 1, 1), dt)
                for i in range(len(new) - 1, -1, -1):
                    S = new[i]
                    Y = np.matmul(S.reshape(len(idx), -1, S.shape[3]), C)
                    Y = Y.reshape(len(idx), S.shape[1], -1)
                    if i:
                        U, s, Vh = np.linalg.svd(Y, full_matrices=False)
                        k = min(chi, s.shape[1])
                        C, V = U[:, :, :k] * s[:, None, :k], Vh[:, :k]
                        f = np.linalg.norm(C, axis=(1, 2), keepdims=True)
                        C, lg = C / f, lg + np.log(f[:, 0, 0])
                    else:
                        V = Y
                    new[i] = V.reshape(len(idx), V.shape[1], S.shape[2], -1)
                M = new
                got.append((M, lg))
            return got

        with ThreadPoolExecutor(os.cpu_count() or 1) as ex:
            parts = list(ex.map(part, [q for q in np.array_split(np.arange(n), min(n, os.cpu_count() or 1))]))
        return [([torch.from_numpy(np.concatenate([p[j][0][x] for p in parts])).cuda() for x in range(len(host[0]))],
                 torch.from_numpy(np.concatenate([p[j][1] for p in parts])).cuda()) for j in range(len(host) + 1)]


def _value(B, rows, T):
    """<B| rows |T> per configuration: columns absorbed left to right."""
    n = B[0].shape[0]
    L = torch.ones((n, 1) + (1,) * len(rows) + (1,), dtype=B[0].dtype, device="cuda")
    for x in range(len(B)):
        if len(rows) == 1:
            X = torch.einsum("nalb,nadc->nlbdc", L, B[x])
            X = torch.einsum("nlbdc,nlrdu->nbcru", X, rows[0][x])
            L = torch.einsum("nbcru,nbue->ncre", X, T[x])
        else:
            X = torch.einsum("naijb,nadc->nijbdc", L, B[x])
            X = torch.einsum("nijbdc,nikdm->njbckm", X, rows[0][x])
            X = torch.einsum("njbckm,njlmu->nbcklu", X, rows[1][x])
            L = torch.einsum("nbcklu,nbue->nckle", X, T[x])
    return L.reshape(n)


def _spent(c):
    """Seconds, about, that exact() takes: the factorisations on the host dominate."""
    m = min(c["chi"], (c["D"] // c["N"]) ** (c["Lx"] // 2)) * (c["D"] // c["N"])
    rows = (1 if c["kind"] == "amplitude" else 2) * c["Ly"]
    return rows * c["Lx"] * (5e-3 + c["n"] / 16 * (2e-5 + 2.8e-8 * m ** 2.5 * (2 if c["cplx"] else 1)))


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind in ("sample", "multi"):
        return None  # a Markov path, not a computed number
    if kind == "sr":
        return _exact_sr(c, seed)
    if _spent(c) > 20:
        return None
    net = _Net(c, seed)
    Lx, Ly = c["Lx"], c["Ly"]
    rows = [net.row(y) for y in range(Ly)]
    Bs = net.boundary(rows[:-1], False)  # Bs[r]: rows below r
    if kind == "amplitude":
        psi = _value(Bs[Ly - 1][0], [rows[Ly - 1]], [torch.ones_like(t[:, :1, :1, :1]) for t in Bs[0][0]])
        out = dict(log_abs=torch.log(psi.abs()) + Bs[Ly - 1][1], phase=torch.angle(psi))
        return out
    Ts = net.boundary(rows[:0:-1], True)[::-1]  # Ts[r]: rows above r
    B, T = [b[0] for b in Bs], [t[0] for t in Ts]
    if kind in ("gradient", "autograd"):
        return _exact_grad(c, seed, net, rows, Bs, T)
    return dict(e_loc=_exact_energy(c, net, rows, B, T))


def _exact_grad(c, seed, net, rows, Bs, T):
    Lx, Ly, D4 = c["Lx"], c["Ly"], net.Dk ** 4
    O = torch.zeros((c["n"], Lx * Ly, D4), dtype=net.theta.dtype, device="cuda")
    bid = torch.stack([net.block(x, y) for y in range(Ly) for x in range(Lx)], 1)
    for y in range(Ly):
        W = [t.detach().clone().requires_grad_() for t in rows[y]]
        val = _value(Bs[y][0], [W], T[y])
        for x, g in enumerate(torch.autograd.grad(val, W, torch.ones_like(val))):
            # d val / d W without conjugation
            g = (g.conj() / val.detach().reshape(-1, 1, 1, 1, 1)).reshape(c["n"], -1)
            O[:, y * Lx + x, :g.shape[1]] = g
    if c["kind"] == "gradient":
        return dict(block_ids=None, O=O)
    psi = _value(Bs[Ly - 1][0], [rows[Ly - 1]], T[Ly - 1])
    w = torch.from_numpy(_rng(seed, 4).standard_normal(c["n"])).cuda()
    grad = torch.zeros(net.off[-1], dtype=torch.float64, device="cuda")
    for v in range(Lx * Ly):
        at = net.off[v] + bid[:, v, None] * net.bs[v] + torch.arange(net.bs[v], device="cuda")
        grad.index_add_(0, at.reshape(-1), (w[:, None] * O[:, v, :net.bs[v]]).reshape(-1))
    return dict(log_abs=torch.log(psi.abs()) + Bs[Ly - 1][1], grad=grad)


def _exact_energy(c, net, rows, B, T):
    Lx, Ly, N = c["Lx"], c["Ly"], c["N"]
    cos = 2.0 - 2.0 * torch.cos(2.0 * math.pi * torch.arange(N, device="cuda", dtype=torch.float64) / N)
    e = COUPLING["g"] * (cos[net.h].sum((1, 2)) + cos[net.v].sum((1, 2))).to(net.theta.dtype)
    J = J_HOP if c["matter"] else 0.0

    def ratio(r, two, den, sites):
        new = [list(rows[r + i]) for i in range(2 if two else 1)]
        for x, y in sites:
            new[y - r][x] = net.tensor(x, y)
        return _value(B[r], new, T[r + (1 if two else 0)]) / den

    def hop(link, a, b, val):
        """Adds J psi(s')/psi(s) of the hop across link (in place while val() runs)."""
        pa, pb, l0 = a.clone(), b.clone(), link.clone()
        d = pb - pa  # +1: the boson comes over the link and raises it
        a += d
        b -= d
        link.copy_((link + d) % N)
        q = val()
        a.copy_(pa)
        b.copy_(pb)
        link.copy_(l0)
        return J * torch.where(d != 0, q, torch.zeros_like(q))

    for r in range(Ly):
        if J:
            den = _value(B[r], [rows[r]], T[r])
            for x in range(Lx - 1):
                e = e + hop(net.h[:, r, x], net.p[:, r, x], net.p[:, r, x + 1],
                            lambda: ratio(r, False, den, [(x, r), (x + 1, r)]))
        if r == Ly - 1:
            break
        den = _value(B[r], [rows[r], rows[r + 1]], T[r + 1])
        for x in range(Lx - 1):
            for t in ((1,) if N == 2 else (1, N - 1)):
                keep = net.h.clone(), net.v.clone()
                net.h[:, r, x] += t
                net.v[:, r, x + 1] += t
                net.h[:, r + 1, x] -= t
                net.v[:, r, x] -= t
                net.h %= N
                net.v %= N
                e = e - (2.0 if N == 2 else 1.0) * COUPLING["h"] * ratio(
                    r, True, den, [(x, r), (x + 1, r), (x, r + 1), (x + 1, r + 1)])
                net.h, net.v = keep
        if J:
            for x in range(Lx):
                e = e + hop(net.v[:, r, x], net.p[:, r, x], net.p[:, r + 1, x],
                            lambda: ratio(r, True, den, [(x, r), (x, r + 1)]))
    return e.to(torch.complex128)


def _exact_sr(c, seed):
    nb, bs, off = _vertex_tables(c)
    s, n, Np = _samples(c, seed), c["n"], off[-1]
    dt = torch.complex128 if c["cplx"] else torch.float64
    O, E = s["O"].to(dt), torch.view_as_complex(s["e_loc"].view(n, 2)).to(torch.complex128)
    at = [off[v] + s["block_ids"][:, v].long()[:, None] * bs[v] + torch.arange(bs[v], device="cuda")
          for v in range(len(nb))]

    def gather(x):
        return sum((O[:, v, :bs[v]] * x[at[v]]).sum(1) for v in range(len(nb)))

    def scatter(t, sq=False):
        out = torch.zeros(Np, dtype=dt, device="cuda")
        for v in range(len(nb)):
            o = O[:, v, :bs[v]]
            out.index_add_(0, at[v].reshape(-1), ((o.abs() ** 2 if sq else o.conj()) * t[:, None]).to(dt).reshape(-1))
        return out

    ones = torch.full((n,), 1.0 / n, dtype=dt, device="cuda")
    Em = E.mean()
    F = scatter(((E - Em) if c["cplx"] else (E - Em).real) / n)
    if n >= Np:
        d = (scatter(ones, True).real - scatter(ones).abs() ** 2).clamp(min=0) + CG["diag_shift"]
    else:
        d = torch.ones(Np, dtype=torch.float64, device="cuda")
    x, r = torch.zeros_like(F), F.clone()
    z = r / d
    p, rz, f = z.clone(), torch.vdot(r, z).real, torch.linalg.norm(F)
    for _ in range(CG["max_iter"]):
        t = gather(p)
        q = scatter((t - t.mean()) / n) + CG["diag_shift"] * p
        a = rz / torch.vdot(p, q).real
        x, r = x + a * p, r - a * q
        z = r / d
        new = torch.vdot(r, z).real
        p, rz = z + (new / rz) * p, new
        if torch.linalg.norm(r) <= CG["tol"] * f:
            break
    A = torch.from_numpy(_tensors(c, seed, Np)).cuda()
    A = A + (0.5 + 0.5j) * 0.01 * (-1j) * x if c["cplx"] else A - 0.01 * x
    err = E.real.std(correction=1) / math.sqrt(n)
    return dict(stats=torch.stack([Em.real, err, f]), tensors=A)
