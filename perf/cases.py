"""The calls a user of the library times: what they are, their inputs, one pass, and its 64-bit value.

Every case is one entry point of the package on one system (grid of k-points, M orbitals and n
occupied orbitals per k, G Cholesky vectors per momentum transfer, W walkers):

  energy          KPointAFQMC.local_energy: Green's function, Cholesky traces, E1, E_C, E_X
  propagate       KPointAFQMC.propagate: force bias, vHS, Taylor series, weight, optional QR
  orthonormalise  KPointAFQMC.orthonormalise
  adjoint         LocalEnergy.apply forward and backward (gradients in the walkers and in h)
  block           KPointAFQMC.block / DenseAFQMC.block: device fields, steps, QR, comb
  group           KPointGroup.step over several uneven systems

Inputs are drawn on the GPU from the seed: Cholesky vectors complex N(0,1) exp(-g/16)/sqrt(Nk M)
with L[-Q, k-Q] = L[Q, k]^dagger, h = diag(0..4) plus a small Hermitian part, walkers the
orthonormalised trial plus 10% noise per column (what a projection that starts from the trial
carries), normal fields.  Calls that update the walkers start each pass from the same ones.
"""
from __future__ import annotations

import itertools
import math

import torch

from paper_2003_09468_gb300 import DenseAFQMC, KPointAFQMC, KPointGroup, LocalEnergy

DT = 0.005
ORDER = 6   # terms of the Taylor series
C128 = torch.complex128

# Eight uneven systems advanced as one group, "grid/M/n/W" each, 8 M vectors per Q.
UNEVEN = ("2x2x2/16/2/256 2x2x2/26/4/128 2x2x3/16/2/160 2x2x3/26/4/96 "
          "2x3x3/16/4/128 2x3x3/26/2/96 3x3x3/16/2/128 3x3x3/26/4/32")


def _case(kind, grid, M, n, G, W, **more):
    return {"kind": kind, "grid": grid, "M": M, "n": n, "G": G, "W": W, "precision": "mixed", "trial": "identity",
            **more}


def listed():
    return [
        # the smallest system of the test suite: launches and latency
        {"name": "energy-2x2x2", **_case("energy", "2x2x2", 8, 2, 48, 16)},
        # the same system on the FP64 path, which users run to check the mixed one
        {"name": "energy-fp64-2x2x2", **_case("energy", "2x2x2", 8, 2, 48, 16, precision="fp64")},
        # odd and ragged sizes, a trial that is not the first n orbitals, a QR in the step
        {"name": "propagate-ragged-3x1x2", **_case("propagate", "3x1x2", 7, 3, 23, 37, trial="random", qr=True)},
        # a Gamma-point supercell in the standard (dense) representation, real vectors
        {"name": "block-dense-1x1x2", **_case("block", "dense", 52, 8, 416, 64, steps=5, qr_period=5,
                                              energy_period=5)},
        # a medium crystal as a production run drives it: several steps per energy
        {"name": "block-2x2x3", **_case("block", "2x2x3", 26, 4, 208, 96, steps=5, qr_period=5, energy_period=5)},
        # the paper's 3x3x3 double-zeta size, one call of each kind
        {"name": "propagate-3x3x3", **_case("propagate", "3x3x3", 26, 4, 208, 64, qr=False)},
        {"name": "energy-3x3x3", **_case("energy", "3x3x3", 26, 4, 208, 64)},
        {"name": "orthonormalise-3x3x3", **_case("orthonormalise", "3x3x3", 26, 4, 208, 64)},
        {"name": "adjoint-3x3x3", **_case("adjoint", "3x3x3", 26, 4, 208, 64)},
        # the benchmark's workload: every step with its energy, a QR every fifth
        {"name": "block-3x3x3", **_case("block", "3x3x3", 26, 4, 208, 64, steps=5, qr_period=5, energy_period=1)},
        # a dense k-mesh in a minimal basis: many k-points, 256 electrons per spin
        {"name": "block-4x4x4", **_case("block", "4x4x4", 8, 4, 64, 32, steps=2, qr_period=2, energy_period=2)},
        # eight uneven systems, 1024 walkers, one step with energies
        {"name": "group-uneven-8", "kind": "group", "members": UNEVEN, "qr": False},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    top = max((work(c) for c in listed()), key=lambda w: w["flops"])
    while True:
        kind = rng.choice(["energy", "propagate", "orthonormalise", "adjoint", "block", "block", "dense", "group"])
        if kind == "group":
            members = []
            for _ in range(rng.randint(2, 4)):
                grid = "x".join(str(rng.randint(1, 3)) for _ in range(3))
                M = _logint(rng, 6, 26)
                members.append("%s/%d/%d/%d" % (grid, M, min(M, _logint(rng, 1, 5)), _logint(rng, 3, 128)))
            c = {"kind": "group", "members": " ".join(members), "qr": rng.random() < 0.5}
        else:
            grid = "dense" if kind == "dense" else "x".join(str(rng.choice([1, 2, 2, 3, 3])) for _ in range(3))
            M = _logint(rng, 4, 52)
            n = min(M, _logint(rng, 1, 8))
            c = _case("block" if kind == "dense" else kind, grid, M, n, max(2, int(M * rng.uniform(3, 9))),
                      _logint(rng, 2, 160), trial=rng.choice(["identity", "random"]))
            if kind == "propagate":
                c["qr"] = rng.random() < 0.5
            if kind in ("block", "dense"):
                c["steps"] = rng.randint(1, 5)
                c["qr_period"] = rng.choice([2, 5])
                c["energy_period"] = rng.randint(1, c["steps"])
            if kind in ("energy", "propagate") and rng.random() < 0.2:
                c["precision"] = "fp64"
        w = work(c)
        fp64 = c.get("precision") == "fp64"
        # the handle's set-up (the exchange tensor's build) no dearer than the 3x3x3 system's either
        setup = sum(_setup(m) for m in (_members(c) if kind == "group" else [c]))
        if (w["flops"] <= (0.004 if fp64 else 1.0) * top["flops"] and w["bytes"] <= top["bytes"]
                and setup <= _setup(_case("energy", "3x3x3", 26, 4, 208, 1))):
            return c


# ------------------------------------------------------------------ sizes and work
def _sizes(c):
    if c["grid"] == "dense":
        grid = (1, 1, 1)
    else:
        grid = tuple(int(v) for v in c["grid"].split("x"))
    return grid, math.prod(grid), c["M"], c["n"], c["G"], c["W"]


def _members(c):
    out = []
    for i, m in enumerate(c["members"].split()):
        grid, M, n, W = m.split("/")
        out.append(_case("step", grid, int(M), int(n), 8 * int(M), int(W)))
    return out


def work(case):
    if case["kind"] == "group":
        ws = [work(dict(m, kind="block", steps=1, qr_period=int(case["qr"]), energy_period=1))
              for m in _members(case)]
        return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}
    _, nk, M, n, G, W = _sizes(case)
    N, NM, ws = nk * n, nk * M, 2 * W
    cb = 16 if case["precision"] == "fp64" else 8   # one complex number of the handle's static data
    phi = 16 * ws * NM * N
    green = 8 * ws * (N * N * M + N ** 3 + N * N * NM)
    half = 8 * W * nk * nk * G * n * M               # the Cholesky traces
    exch = 8 * ws * (nk ** 3 / 2) * (n * M) ** 2     # one bilinear form per pair of triples
    lh, z, lv = cb * nk * nk * G * n * M, cb * (nk ** 3 / 2) * (n * M) ** 2, cb * nk * nk * G * M * M
    vhs = 8 * W * nk * nk * G * M * M
    taylor = 8 * ORDER * W * NM * NM * 2 * N + 2 * 8 * ws * nk * M * M * N
    qr = 2 * 8 * ws * NM * N * N
    x = 8 * W * 2 * nk * G
    kind = case["kind"]
    if kind == "energy":
        return {"bytes": phi + lh + z + 48 * W, "flops": green + half + exch}
    if kind == "propagate":
        return {"bytes": 2 * phi + lh + lv + x, "flops": green + half + vhs + taylor + 8 * ws * N ** 3 / 3
                + (qr if case["qr"] else 0)}
    if kind == "orthonormalise":
        return {"bytes": 2 * phi, "flops": qr}
    if kind == "adjoint":
        return {"bytes": 2 * phi + lh + 2 * z + 96 * W, "flops": green + half + 3 * exch + 2 * 8 * ws * N * N * NM}
    steps = case["steps"]
    nqr = -(-steps // case["qr_period"]) if case["qr_period"] else 0
    nen = -(-steps // case["energy_period"])
    # the Green's function of a step's new walkers serves the next step
    return {"bytes": 2 * phi + steps * (lh + lv) + nen * z + 16 * W * steps,
            "flops": (steps + 1) * (green + half) + steps * (vhs + taylor) + nen * exch + nqr * qr}


def _setup(c):
    _, nk, M, n, G, _ = _sizes(c)
    return nk ** 3 * (n * M) ** 2 * G


# ------------------------------------------------------------------ inputs
def _cn(g, *shape):
    return torch.view_as_complex(torch.randn(*shape, 2, generator=g, device="cuda", dtype=torch.float64)) * math.sqrt(0.5)


def _tables(grid):
    k = list(itertools.product(*[range(v) for v in grid]))
    at = {v: i for i, v in enumerate(k)}

    def diff(a, b):
        return at[tuple((x - y) % m for x, y, m in zip(a, b, grid))]

    kminus = [[diff(a, q) for q in k] for a in k]
    return kminus, [diff(k[0], q) for q in k]


def _hermitian(g, nk, M, real):
    r = 0.1 * (torch.randn(nk, M, M, generator=g, device="cuda", dtype=torch.float64).to(C128) if real
               else _cn(g, nk, M, M))
    r = 0.5 * (r + r.mH)
    d = torch.diagonal(r, dim1=-2, dim2=-1)
    d.copy_(torch.linspace(0.0, 4.0, M, device="cuda", dtype=torch.float64).to(C128).expand(nk, M))
    return r


def _system(case, seed):
    """(grid, L, h1, A, phi, g): the Hamiltonian, the trial and the walkers of one case."""
    grid, nk, M, n, G, W = _sizes(case)
    g = torch.Generator("cuda").manual_seed(seed)
    if case["grid"] == "dense":
        L = torch.randn(G, M, M, generator=g, device="cuda", dtype=torch.float64)
        L = (0.5 * (L + L.mT) * torch.exp(-torch.arange(G, device="cuda", dtype=torch.float64) / (2 * M))[:, None, None]
             / math.sqrt(M)).to(C128)
    else:
        L = _cn(g, nk * nk, G, M, M)
        L *= (torch.exp(-torch.arange(G, device="cuda", dtype=torch.float64) / 16) / math.sqrt(nk * M))[:, None, None]
        kminus, minus = _tables(grid)
        first, second = [], []
        for Q in range(nk):
            for k in range(nk):
                b, p = Q * nk + k, minus[Q] * nk + kminus[k][Q]
                if b <= p:
                    first.append(b)
                    second.append(p)
        for i in range(0, len(first), 64):
            a, b = first[i:i + 64], second[i:i + 64]
            own = torch.tensor([x == y for x, y in zip(a, b)], device="cuda")[:, None, None, None]
            blk = L[a]
            blk = torch.where(own, 0.5 * (blk + blk.mH), blk)
            L[a] = blk
            L[b] = blk.mH
        L = L.view(nk, nk, G, M, M)
    h1 = _hermitian(g, nk, M, case["grid"] == "dense")
    if case["trial"] == "random":
        A = torch.linalg.qr(_cn(g, nk, M, M))[0][:, :, :n].contiguous()
    else:
        A = torch.eye(M, n, device="cuda", dtype=C128).expand(nk, M, n).contiguous()
    phi = _cn(g, W, 2, nk * M, nk * n) * (0.1 / math.sqrt(nk * M))
    for k in range(nk):
        phi[:, :, k * M:(k + 1) * M, k * n:(k + 1) * n] += A[k]
    R = torch.linalg.cholesky(phi.mH @ phi).mH
    phi = torch.linalg.solve_triangular(R, phi, upper=True, left=False).contiguous()
    return grid, L, h1, A, phi, g


def _handle(case, grid, L, h1, A):
    if case["grid"] == "dense":
        return DenseAFQMC(L, h1[0], A[0], case["W"], DT, taylor_order=ORDER, precision=case["precision"],
                          hermitian=True)
    return KPointAFQMC(grid, L, h1, A, case["W"], DT, taylor_order=ORDER, precision=case["precision"])


def _fields(case, g, W, nk, G):
    return torch.randn(W, 2, nk, G, generator=g, device="cuda", dtype=torch.float64)


def _own(case, seed):
    grid, L, h1, A, phi, g = _system(case, seed)
    _, nk, M, n, G, W = _sizes(case)
    s = {"case": case, "sys": _handle(case, grid, L, h1, A), "phi0": phi, "seed": seed}
    if case["kind"] in ("propagate", "block", "step"):
        s["phi"] = torch.empty_like(phi)
        s["weight"] = torch.ones(W, device="cuda", dtype=torch.float64)
        s["logdet"] = torch.empty(W, 2, device="cuda", dtype=C128)
        s["x"] = _fields(case, g, W, nk, G)
    if case["kind"] == "orthonormalise":
        # walkers a few steps after their last QR: columns neither orthogonal nor normalised
        s["phi0"] = (phi @ (torch.eye(phi.shape[-1], device="cuda", dtype=C128)
                            + 0.05 * _cn(g, W, 2, phi.shape[-1], phi.shape[-1]) / math.sqrt(phi.shape[-1])))
        s["phi"] = torch.empty_like(phi)
        s["logdet"] = torch.empty(W, 2, device="cuda", dtype=C128)
    if case["kind"] == "adjoint":
        s["h1"] = h1
        s["g"] = _cn(g, W, 3)
    if case["kind"] == "step":
        s["eloc"] = torch.empty(W, 3, device="cuda", dtype=C128)
    if case["kind"] == "block":
        meas = -(-case["steps"] // case["energy_period"])
        s["eloc"] = torch.empty(meas, W, 3, device="cuda", dtype=C128)
        s["weights"] = torch.empty(case["steps"], W, device="cuda", dtype=torch.float64)
        s["counter"] = torch.zeros(1, device="cuda", dtype=torch.int64)
        s["idx"] = torch.empty(W, device="cuda", dtype=torch.int32)
    return s


def prepare(case, seed):
    if case["kind"] == "group":
        parts = [_own(m, seed + 1000 * i) for i, m in enumerate(_members(case))]
        return {"case": case, "parts": parts, "group": KPointGroup([p["sys"] for p in parts])}
    return _own(case, seed)


# ------------------------------------------------------------------ one pass
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "group":
        parts = state["parts"]
        for p in parts:
            p["phi"].copy_(p["phi0"])
            p["weight"].fill_(1.0)
        state["group"].step([p["phi"] for p in parts], [p["x"] for p in parts], [p["weight"] for p in parts],
                            [p["eloc"] for p in parts], [p["logdet"] for p in parts], do_qr=case["qr"], reuse=False)
        return [{k: p[k] for k in ("phi", "weight", "eloc", "logdet")} for p in parts]
    sys = state["sys"]
    if kind == "energy":
        return sys.local_energy(state["phi0"])
    if kind == "adjoint":
        phi, h1 = state["phi0"].requires_grad_(), state["h1"].requires_grad_()
        e = LocalEnergy.apply(phi, h1, sys)
        gphi, gh1 = torch.autograd.grad(e, (phi, h1), state["g"])
        return {"e": e, "grad_phi": gphi, "grad_h1": gh1}
    state["phi"].copy_(state["phi0"])
    if kind == "orthonormalise":
        sys.orthonormalise(state["phi"], state["logdet"])
        return {"phi": state["phi"], "logdet": state["logdet"]}
    state["weight"].fill_(1.0)
    if kind == "propagate":
        sys.propagate(state["phi"], state["x"], state["weight"], state["logdet"], do_qr=case["qr"])
        return {k: state[k] for k in ("phi", "weight", "logdet")}
    state["counter"].zero_()
    sys.block(state["phi"], state["weight"], state["x"], state["eloc"], state["counter"], state["seed"],
              nsteps=case["steps"], qr_period=case["qr_period"], energy_period=case["energy_period"],
              weight_hist=state["weights"], logdet=state["logdet"], comb=True, reuse=False, idx=state["idx"])
    return {k: state[k] for k in ("phi", "weight", "logdet", "eloc", "weights", "idx")}


# ------------------------------------------------------------------ the same in 64 bits
class _Exact:
    """The walker step and the local energy in complex128 PyTorch."""

    def __init__(self, case, seed):
        self.grid, L, self.h1, self.A, self.phi, self.g = _system(case, seed)
        _, self.nk, self.M, self.n, self.G, self.W = _sizes(case)
        if case["grid"] == "dense":
            L = L.view(1, 1, self.G, self.M, self.M)
        kminus, minus = _tables(self.grid)
        self.km = torch.tensor(kminus, device="cuda")
        self.mi = torch.tensor(minus, device="cuda")
        self.L = L
        self.LH = torch.einsum("kpa,qkgpr->qkgar", self.A.conj(), L)

    def green(self, phi):
        W, nk, M, n = phi.shape[0], self.nk, self.M, self.n
        S = torch.einsum("kpa,wskpj->wskaj", self.A.conj(), phi.view(W, 2, nk, M, nk * n)).reshape(W, 2, nk * n, nk * n)
        return torch.linalg.solve(S.mT, phi.mT), S     # [W][2][N][NM]

    def logdet(self, S):
        sign, mag = torch.linalg.slogdet(S)
        return torch.complex(mag, torch.angle(sign))

    def traces(self, Gh):
        W, nk, M, n = Gh.shape[0], self.nk, self.M, self.n
        Gs = Gh.sum(1).view(W, nk, n, nk, M)
        rng = torch.arange(nk, device="cuda")
        X = [torch.einsum("wkar,kgar->wg", Gs[:, rng, :, self.km[:, Q], :].permute(1, 0, 2, 3), self.LH[Q])
             for Q in range(nk)]
        return torch.stack(X, 1)                        # [W][Q][g]

    def xbar(self, X):
        Xm = X[:, self.mi]
        return -math.sqrt(DT) * torch.stack([0.5j * (X + Xm), -0.5 * (X - Xm)], 1)

    def energies(self, Gh, h1, Qs=None):
        """(E1, EC, [E_X of each momentum transfer as a function])."""
        W, nk, M, n = Gh.shape[0], self.nk, self.M, self.n
        G5 = Gh.view(W, 2, nk, n, nk, M)
        Ah = torch.einsum("kpa,kpq->kaq", self.A.conj(), h1)
        e1 = torch.einsum("wskakq,kaq->w", G5, Ah)
        X = self.traces(Gh)
        ec = 0.5 * (X * X[:, self.mi]).sum((1, 2))

        def ex(Q, G5):
            mQ = int(self.mi[Q])
            Z = torch.einsum("kgar,xgbs->kxbras", self.LH[Q], self.LH[mQ]).reshape(nk, nk, n * M, n * M)
            al = G5[:, :, :, :, self.km[:, Q], :].permute(4, 2, 0, 1, 3, 5).reshape(nk, nk, 2 * W, n * M)  # k,x,ws,(b r)
            be = G5[:, :, :, :, self.km[:, mQ], :].permute(2, 4, 0, 1, 3, 5).reshape(nk, nk, 2 * W, n * M)  # k,x,ws,(a s)
            return -0.5 * ((al @ Z) * be).sum((0, 1, 3)).view(W, 2).sum(1)

        return e1, ec, ex, G5

    def local_energy(self, phi):
        Gh, _ = self.green(phi)
        e1, ec, ex, G5 = self.energies(Gh, self.h1)
        return torch.stack([e1, ec, sum(ex(Q, G5) for Q in range(self.nk))], 1)

    def propagate(self, phi, x):
        W, nk, M = phi.shape[0], self.nk, self.M
        Gh, S = self.green(phi)
        xb = self.xbar(self.traces(Gh))
        xt = x - xb
        y = 0.5 * (1j * xt[:, 0] - xt[:, 1]) + 0.5 * (1j * xt[:, 0][:, self.mi] + xt[:, 1][:, self.mi])
        V = torch.zeros(W, nk, M, nk, M, device="cuda", dtype=C128)
        rng = torch.arange(nk, device="cuda")
        v0 = torch.zeros(nk, M, M, device="cuda", dtype=C128)
        for Q in range(nk):
            V[:, rng, :, self.km[:, Q], :] = math.sqrt(DT) * torch.einsum("wg,kgpr->kwpr", y[:, Q], self.L[Q])
            v0 -= 0.5 * torch.einsum("kgpr,kgqr->kpq", self.L[Q], self.L[Q].conj())
        V = V.view(W, 1, nk * M, nk * M)
        E = torch.linalg.matrix_exp(-0.5 * DT * (self.h1 + v0))

        def half(u):
            return (E @ u.view(W, 2, nk, M, -1)).view(u.shape)

        acc = term = half(phi)
        for j in range(1, ORDER + 1):
            term = (V @ term) / j
            acc = acc + term
        new = half(acc)
        _, Sn = self.green(new)
        old, ld = self.logdet(S), self.logdet(Sn)
        d = (ld - old).sum(1)
        logi = d + (x * xb - 0.5 * xb * xb).sum((1, 2, 3))
        return new, torch.exp(logi.real) * torch.cos(d.imag).clamp_min(0.0), ld

    def qr(self, phi):
        Q, R = torch.linalg.qr(phi)
        d = torch.diagonal(R, dim1=-2, dim2=-1)
        Q = Q * (d / d.abs()).unsqueeze(-2)
        return Q, self.logdet(self.green(Q)[1])


def exact(case, seed):
    if case["kind"] in ("block", "group"):
        return None   # several steps, fields drawn on the device
    if case["kind"] == "orthonormalise":
        e = _Exact(case, seed)
        N = e.phi.shape[-1]
        phi = e.phi @ (torch.eye(N, device="cuda", dtype=C128)
                       + 0.05 * _cn(e.g, case["W"], 2, N, N) / math.sqrt(N))
        return dict(zip(("phi", "logdet"), e.qr(phi)))
    e = _Exact(case, seed)
    if case["kind"] == "energy":
        return e.local_energy(e.phi)
    if case["kind"] == "propagate":
        x = _fields(case, e.g, e.W, e.nk, e.G)
        phi, weight, ld = e.propagate(e.phi, x)
        if case["qr"]:
            phi, ld = e.qr(phi)
        return {"phi": phi, "weight": weight, "logdet": ld}
    g = _cn(e.g, e.W, 3)
    phi, h1 = e.phi.requires_grad_(), e.h1.requires_grad_()
    Gh, _ = e.green(phi)
    leaf = Gh.detach().requires_grad_()
    e1, ec, ex, _ = e.energies(leaf, h1)
    gh1, gG = torch.autograd.grad([e1, ec], (h1, leaf), [g[:, 0].contiguous(), g[:, 1].contiguous()])
    tot = torch.zeros_like(ec)
    for Q in range(e.nk):   # one momentum transfer at a time: the intermediates of all do not fit
        q = ex(Q, leaf.view(e.W, 2, e.nk, e.n, e.nk, e.M))
        gG = gG + torch.autograd.grad(q, leaf, g[:, 2].contiguous())[0]
        tot = tot + q.detach()
    gphi = torch.autograd.grad(Gh, phi, gG)[0]
    return {"e": torch.stack([e1.detach(), ec.detach(), tot], 1), "grad_phi": gphi, "grad_h1": gh1}
