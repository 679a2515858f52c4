"""The measured work: what programs that use this package have it do, through
its public entry points (WilsonDirac, WilsonBatch, Krylov, PtcNet, Fgcr).

Lattices, hopping parameters, sources and solver settings are those of the
seeded workloads (``synthetic/workloads.py``), of ``bench.py`` and of the tests;
the gauge fields are the same kind of field (U = exp(i eps H), eps = 0.3),
drawn on the GPU.  Boundary phases: periodic in space, antiperiodic in time.
"""
from __future__ import annotations

import math

import torch

from paper_1401_2039_gb300 import Fgcr, Krylov, PtcNet, WilsonBatch, WilsonDirac
from paper_1401_2039_gb300.train_preconditioner import neumann_weights

PHASE = (1.0, 1.0, 1.0, -1.0)
EPS = 0.3
CHANNELS = (1, 16, 16, 16, 1)
BYTES = {"f64": 8, "f32": 4, "f16": 2, "bf16": 2}
TOL = 1e-10


def _dims(text: str) -> tuple:
    return tuple(int(v) for v in text.split("x"))


def _lattices(case) -> list:
    return [_dims(t) for t in case["dims"].split("+")]


def _volume(dims) -> int:
    return dims[0] * dims[1] * dims[2] * dims[3]


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # The benchmark's solve: one Gaussian source on the large lattice in half-precision
        # storage with 12-real links, defect correction to a 1e-10 true residual.
        {"name": "solve_f16r12_large", "kind": "solve", "dims": "32x32x32x64", "prec": "f16",
         "recon": 12, "kappa": 0.124, "recovery": "defect", "inner": 1e-3, "mu": 0.0},
        # The mixed-precision solve with the handle's defaults (FP32 storage, reliable
        # updates) on a lattice whose fields stay in L2.
        {"name": "solve_f32_medium", "kind": "solve", "dims": "16x16x16x32", "prec": "f32",
         "recon": 18, "kappa": 0.124, "recovery": "reliable", "inner": 0.1, "mu": 0.0},
        # The plain FP64 solve of the package's default precision on the paper's lattice: what
        # every faster solve is compared with.
        {"name": "solve_f64_paper", "kind": "solve", "dims": "24x24x24x48", "prec": "f64",
         "recon": 18, "kappa": 0.12, "recovery": "reliable", "inner": 0.1, "mu": 0.0},
        # The smallest workload: a solve that is all latency.
        {"name": "solve_f64_small", "kind": "solve", "dims": "4x4x4x4", "prec": "f64",
         "recon": 18, "kappa": 0.12, "recovery": "reliable", "inner": 0.1, "mu": 0.0},
        # A quark propagator: the twelve spin-colour point sources of one site as one batch.
        {"name": "batch_propagator", "kind": "batch", "dims": "24x24x24x48", "nrhs": 12,
         "prec": "f32", "recon": 18, "kappa": 0.12, "recovery": "defect", "inner": 1e-5,
         "source": "point"},
        # A serving batch: four sources on each of three lattices of different sizes.
        {"name": "batch_uneven", "kind": "batch", "dims": "8x8x8x8+12x12x12x24+16x16x16x32",
         "nrhs": 4, "prec": "f32", "recon": 18, "kappa": 0.12, "recovery": "reliable",
         "inner": 0.1, "source": "gaussian"},
        # The full operator in FP64 (residual checks, measurements on solutions).
        {"name": "apply_f64_paper", "kind": "apply", "dims": "24x24x24x48", "prec": "f64",
         "recon": 18, "kappa": 0.12, "dagger": False, "mu": 0.0},
        # The even-odd operator and its adjoint inside a caller's own solver: BF16 storage on an
        # anisotropic lattice with ragged last blocks and a twisted mass.
        {"name": "schur_bf16_ragged", "kind": "apply_eo", "dims": "28x20x36x46", "prec": "bf16",
         "recon": 18, "kappa": 0.124, "dagger": True, "mu": 0.05, "parity": 0},
        # One hopping term on a small odd-shaped lattice: mostly launches.
        {"name": "hop_f32r12_tiny", "kind": "dslash_eo", "dims": "6x10x14x18", "prec": "f32",
         "recon": 12, "kappa": 0.12, "dagger": False, "mu": 0.0, "parity": 1},
        # The solver comparison's conjugate residual in FP64.
        {"name": "krylov_mcr2", "kind": "krylov", "dims": "16x16x16x32", "method": "mcr2",
         "kappa": 0.12},
        # One application of the learned preconditioner's network on its training lattice.
        {"name": "net_apply", "kind": "net", "dims": "16x16x16x32", "kappa": 0.124},
        # The gradient of its training loss (forward and backward) on a minibatch.
        {"name": "net_gradient", "kind": "grad", "dims": "8x8x8x16", "samples": 4,
         "kappa": 0.124},
    ]


def _draw_dims(rng, lo: int, hi: int) -> str:
    """Four even extents, 2 .. 64, of a volume between about lo and hi, spread
    over its logarithm."""
    while True:
        v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        d = [max(2, 2 * round(0.5 * v ** 0.25 * math.exp(rng.uniform(-0.45, 0.45))))
             for _ in range(4)]
        d[3] = max(2, 2 * round(0.5 * v / (d[0] * d[1] * d[2])))
        if max(d) <= 64 and lo <= _volume(d) <= hi:
            return "x".join(str(x) for x in d)


def draw(rng):
    kind = rng.choice(["apply", "apply_eo", "dslash_eo", "solve", "solve", "solve", "solve",
                       "batch", "batch", "krylov", "net", "grad", "fgcr"])
    kappa = rng.choice([0.115, 0.12, 0.124])
    prec = rng.choice(["f64", "f64", "f32", "f32", "f16", "f16", "bf16"])
    recon = rng.choice([18, 18, 12])
    if kind in ("apply", "apply_eo", "dslash_eo"):
        c = {"kind": kind, "dims": _draw_dims(rng, 2 ** 8, 2 ** 21), "prec": prec, "recon": recon,
             "kappa": kappa, "dagger": rng.random() < 0.5,
             "mu": rng.choice([0.0, 0.0, 0.05]) if kind != "dslash_eo" else 0.0}
        if kind != "apply":
            c["parity"] = rng.randint(0, 1)
        return c
    recovery, inner = rng.choice([("reliable", 0.1), ("defect", 0.01), ("defect", 1e-3)])
    if kind == "solve":
        # the FP64 solve costs the most: at most the paper's lattice
        top = 600000 if prec == "f64" else 2 ** 21
        return {"kind": kind, "dims": _draw_dims(rng, 2 ** 8, top), "prec": prec, "recon": recon,
                "kappa": kappa, "recovery": recovery, "inner": inner,
                "mu": rng.choice([0.0, 0.0, 0.05])}
    if kind == "batch":
        n = rng.randint(1, 3)
        return {"kind": kind, "dims": "+".join(_draw_dims(rng, 2 ** 9, 2 ** 18) for _ in range(n)),
                "nrhs": rng.randint(1, 12), "prec": rng.choice(["f32", "f32", "f16"]),
                "recon": recon, "kappa": kappa, "recovery": recovery, "inner": inner,
                "source": rng.choice(["gaussian", "point"])}
    if kind == "krylov":
        return {"kind": kind, "dims": _draw_dims(rng, 2 ** 9, 2 ** 17),
                "method": rng.choice(["cgnr", "crne", "mcr1", "mcr2"]), "kappa": kappa}
    if kind == "net":
        return {"kind": kind, "dims": _draw_dims(rng, 2 ** 9, 2 ** 18), "kappa": kappa}
    if kind == "grad":
        return {"kind": kind, "dims": _draw_dims(rng, 2 ** 9, 2 ** 15),
                "samples": rng.randint(1, 6), "kappa": kappa}
    return {"kind": kind, "dims": _draw_dims(rng, 2 ** 10, 2 ** 17), "kappa": kappa}


# ------------------------------------------------------------------ inputs
_LAMBDA = None


def _gell_mann_halves():
    """The eight generators lambda_a / 2 as one real-linear map from c_a to H."""
    global _LAMBDA
    if _LAMBDA is None:
        lam = torch.zeros((8, 3, 3), dtype=torch.complex128)
        lam[0, 0, 1] = lam[0, 1, 0] = 1
        lam[1, 0, 1], lam[1, 1, 0] = -1j, 1j
        lam[2, 0, 0], lam[2, 1, 1] = 1, -1
        lam[3, 0, 2] = lam[3, 2, 0] = 1
        lam[4, 0, 2], lam[4, 2, 0] = -1j, 1j
        lam[5, 1, 2] = lam[5, 2, 1] = 1
        lam[6, 1, 2], lam[6, 2, 1] = -1j, 1j
        lam[7, 0, 0] = lam[7, 1, 1] = 1 / math.sqrt(3)
        lam[7, 2, 2] = -2 / math.sqrt(3)
        _LAMBDA = (lam / 2).reshape(8, 9)
    return _LAMBDA


def _mm(a, b):
    """Products of 3x3 matrices stored [3, 3, n]."""
    return torch.stack([torch.stack([a[i, 0] * b[0, k] + a[i, 1] * b[1, k] + a[i, 2] * b[2, k]
                                     for k in range(3)]) for i in range(3)])


def _links(dims, gen):
    """U = exp(i EPS sum_a c_a lambda_a / 2), c_a normal, re-unitarised: [V, 4, 3, 3]."""
    n = 4 * _volume(dims)
    out = torch.empty((n, 3, 3), dtype=torch.complex128, device="cuda")
    lam = _gell_mann_halves().cuda()
    for a in range(0, n, 1 << 20):
        m = min(1 << 20, n - a)
        c = torch.randn((m, 8), generator=gen, device="cuda", dtype=torch.float64)
        X = (c.to(torch.complex128) @ lam).T.reshape(3, 3, m) * (1j * EPS / 4)
        E = torch.zeros_like(X)
        for i in range(3):
            E[i, i] = 1
        T = E
        for k in range(1, 8):
            T = _mm(T, X) / k
            E = E + T
        E = _mm(E, E)
        E = _mm(E, E)
        r0 = E[0] / E[0].abs().square().sum(0).sqrt()
        r1 = E[1] - (r0.conj() * E[1]).sum(0) * r0
        r1 = r1 / r1.abs().square().sum(0).sqrt()
        r2 = torch.stack([r0[1] * r1[2] - r0[2] * r1[1], r0[2] * r1[0] - r0[0] * r1[2],
                          r0[0] * r1[1] - r0[1] * r1[0]]).conj()
        out[a:a + m] = torch.stack([r0, r1, r2]).permute(2, 0, 1)
    return out.reshape(n // 4, 4, 3, 3)


def _gaussian(shape, gen):
    re = torch.randn(shape, generator=gen, device="cuda", dtype=torch.float64)
    im = torch.randn(shape, generator=gen, device="cuda", dtype=torch.float64)
    return torch.complex(re, im) * math.sqrt(0.5)


def _inputs(case, seed):
    """(links, right-hand sides or fields) of every lattice of the case, from the seed."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed) * 7919 + 17)
    Us, fs = [], []
    for dims in _lattices(case):
        V = _volume(dims)
        Us.append(_links(dims, gen))
        kind = case["kind"]
        if kind in ("apply_eo", "dslash_eo"):
            fs.append(_gaussian((V // 2, 3, 4), gen))
        elif kind == "batch":
            n = case["nrhs"]
            if case["source"] == "gaussian":
                fs.append(_gaussian((n, V, 3, 4), gen))
            else:   # the spin-colour unit sources of one site
                b = torch.zeros((n, V, 3, 4), dtype=torch.complex128, device="cuda")
                site = int(torch.randint(V, (1,), generator=gen, device="cuda"))
                for k in range(n):
                    b[k, site, (k // 4) % 3, k % 4] = 1
                fs.append(b)
        elif kind == "grad":
            fs.append(_gaussian((case["samples"], V, 3, 4), gen))
        else:
            fs.append(_gaussian((V, 3, 4), gen))
    return Us, fs


def _weights(case, seed):
    """The network at its hand-built start (degree-4 Neumann polynomial, small noise)."""
    return torch.from_numpy(neumann_weights(CHANNELS, case["kappa"], int(seed))).cuda()


def _operator(case, dims, U, prec, recon=18):
    op = WilsonDirac(dims, case["kappa"], PHASE, prec=prec, recon=recon)
    op.set_gauge(U)
    if case.get("recovery"):
        op.set_recovery(case["recovery"], case["inner"])
    if case.get("mu"):
        op.set_twisted_mass(case["mu"])
    return op


def prepare(case, seed):
    kind = case["kind"]
    Us, fs = _inputs(case, seed)
    dims = _lattices(case)
    st = {"kind": kind, "case": case, "in": fs[0]}
    if kind == "batch":
        st["ops"] = [_operator(case, d, U, case["prec"], case["recon"]) for d, U in zip(dims, Us)]
        st["batch"] = WilsonBatch(st["ops"], [case["nrhs"]] * len(dims))
        st["in"] = fs
    elif kind in ("net", "grad"):
        st["net"] = PtcNet(dims[0], PHASE, CHANNELS)
        st["net"].set_gauge(Us[0])
        st["net"].set_weights(_weights(case, seed))
        if kind == "grad":   # training pairs: e and r = D e
            op = _operator(case, dims[0], Us[0], "f64")
            st["e"] = fs[0]
            st["in"] = torch.stack([op.apply(e) for e in fs[0]])
            torch.cuda.synchronize()
    elif kind == "fgcr":
        st["lo"] = _operator(case, dims[0], Us[0], "f32")
        st["hi"] = _operator(case, dims[0], Us[0], "f64")
        st["net"] = PtcNet(dims[0], PHASE, CHANNELS)
        st["net"].set_gauge(Us[0])
        st["net"].set_weights(_weights(case, seed))
        st["fgcr"] = Fgcr(st["lo"], st["hi"], st["net"], 16)
    elif kind == "krylov":
        st["op"] = _operator(case, dims[0], Us[0], "f64")
        st["krylov"] = Krylov(st["op"], case["method"])
    else:
        st["op"] = _operator(case, dims[0], Us[0], case["prec"], case["recon"])
    return st


def run(st):
    kind, case = st["kind"], st["case"]
    if kind == "solve":
        return st["op"].solve(st["in"], tol=TOL).x
    if kind == "batch":
        return st["batch"].solve(st["in"], tol=TOL)[0]
    if kind == "apply":
        return st["op"].apply(st["in"], dagger=case["dagger"])
    if kind == "apply_eo":
        return st["op"].apply_eo(st["in"], parity=case["parity"], dagger=case["dagger"])
    if kind == "dslash_eo":
        return st["op"].dslash_eo(st["in"], case["parity"], dagger=case["dagger"])
    if kind == "krylov":
        return st["krylov"].solve(st["in"], tol=TOL).x
    if kind == "net":
        return st["net"].apply(st["in"])
    if kind == "grad":
        loss, grad = st["net"].loss_grad(st["in"], st["e"])
        return {"loss": loss, "grad": grad}
    return st["fgcr"].solve(st["in"], tol=TOL).x


# ------------------------------------------------------------------ work
HOP_FLOPS = 1320     # one hopping term per output site


def work(case):
    """Bytes and operations that the path cannot do without: fields in and
    out once in the caller's complex128, links once in the storage precision.
    A solve adds the iterations that this kind of field needs at its kappa
    (measured once with plain FP64 CGNR), each with its hopping terms and
    vector updates in the storage precision."""
    kind = case["kind"]
    prec, recon = case.get("prec", "f64"), case.get("recon", 18)
    s = BYTES[prec]
    V = sum(_volume(d) for d in _lattices(case))
    if kind == "net" or kind == "grad":
        n = case.get("samples", 1)
        mac = sum(a * b for a, b in zip(CHANNELS, CHANNELS[1:])) * 9 * 16 * 3
        hops = sum(CHANNELS[:-1]) * 8 * 36
        passes = 1 if kind == "net" else 3
        return {"bytes": V * (4 * 18 * 4 + 192 * (2 if kind == "net" else 2 * n)),
                "flops": 8.0 * V * n * passes * (mac + hops)}
    if kind == "apply":
        return {"bytes": V * (2 * 192 + 4 * recon * s), "flops": V * (HOP_FLOPS + 48.0)}
    if kind in ("apply_eo", "dslash_eo"):
        hops = 2 if kind == "apply_eo" else 1
        return {"bytes": V // 2 * 2 * 192 + V * 4 * recon * s,
                "flops": V / 2 * (hops * HOP_FLOPS + 48.0)}
    n = case.get("nrhs", 1)
    iters = {0.115: 60, 0.12: 70, 0.124: 95}[case["kappa"]]
    hop = V / 2 * (48 * n + 8 * recon) * s
    field = V / 2 * 24 * s * n
    if kind == "krylov":   # one (mcr2) or two Schur operators an iteration
        its = iters * (2 if case["method"].startswith("mcr") else 1)
        per = 2 if case["method"] == "mcr2" else 4
        return {"bytes": its * (per * hop + 10 * field) + 2 * 192 * V,
                "flops": its * per * V / 2 * (HOP_FLOPS + 48.0)}
    if kind == "fgcr":     # about 45 directions, each a network application and an operator
        net = work({"kind": "net", "dims": case["dims"]})
        return {"bytes": 45 * (net["bytes"] + 2 * hop / 2 + 16 * 192 * V),
                "flops": 45 * (net["flops"] + V * (HOP_FLOPS + 48.0))}
    return {"bytes": iters * (4 * hop + 2 * field + 8 * field) + 2 * 192 * V * n,
            "flops": iters * 4 * V / 2 * (HOP_FLOPS + 48.0) * n}


# ------------------------------------------------------------------ exact values
# DeGrand-Rossi gamma matrices: row s has its one entry coef[s] in column col[s]
_GAMMA = (((3, 2, 1, 0), (1j, 1j, -1j, -1j)), ((3, 2, 1, 0), (-1, 1, 1, -1)),
          ((2, 3, 0, 1), (1j, -1j, -1j, 1j)), ((2, 3, 0, 1), (1, 1, 1, 1)))


class _Plain:
    """Transports and the Wilson-Dirac operator in plain torch on fields
    [n, T, Z, Y, X, 3, S] (n fields on one gauge field)."""

    def __init__(self, dims, U, dtype):
        self.shape = tuple(reversed(dims))
        self.U = [U[:, m].reshape(self.shape + (3, 3)).to(dtype) for m in range(4)]
        self.gamma = [(list(c), torch.tensor(v, dtype=dtype, device="cuda")) for c, v in _GAMMA]
        self.dtype = dtype

    def field(self, psi):
        return psi.reshape((-1,) + self.shape + psi.shape[-2:]).to(self.dtype)

    def transport(self, psi, mu, forward):
        ax = 4 - mu
        U = self.U[mu]
        if forward:
            f = torch.roll(psi, -1, ax)
            f.select(ax, self.shape[3 - mu] - 1).mul_(PHASE[mu])
            return sum(U[..., :, b, None] * f[..., b, None, :] for b in range(3))
        g = sum(U[..., b, :, None].conj() * psi[..., b, None, :] for b in range(3))
        g = torch.roll(g, 1, ax)
        g.select(ax, 0).mul_(PHASE[mu])
        return g

    def spin(self, mu, t):
        col, coef = self.gamma[mu]
        return t[..., col] * coef

    def hop(self, psi, dagger=False):
        out = torch.zeros_like(psi)
        for mu in range(4):
            for fwd in (True, False):
                t = self.transport(psi, mu, fwd)
                out += t
                out.add_(self.spin(mu, t), alpha=-1 if fwd != dagger else 1)
        return out

    def twist(self, psi, t):   # (1 + i t gamma5) psi
        if t == 0.0:
            return psi
        d = torch.tensor([1 + 1j * t, 1 + 1j * t, 1 - 1j * t, 1 - 1j * t], dtype=self.dtype,
                         device="cuda")
        return psi * d

    def dirac(self, psi, kappa, mu=0.0, dagger=False):
        t = 2 * kappa * mu * (-1 if dagger else 1)
        return self.twist(psi, t) - kappa * self.hop(psi, dagger)


def _dot(a, b):
    return (a.conj() * b).flatten(1).sum(1).reshape(-1, 1, 1, 1, 1, 1, 1)


def _inner(P, r, kappa, mu, steps=40, tol=1e-3):
    """BiCGStab on n systems at once from 0, until every residual fell by tol."""
    x = torch.zeros_like(r)
    r0, p, v = r.clone(), torch.zeros_like(r), torch.zeros_like(r)
    rho = alpha = om = torch.ones_like(_dot(r, r))
    n0 = _dot(r, r).real
    tiny = 1e-30
    for k in range(steps):
        rho1 = _dot(r0, r)
        beta = (rho1 / (rho + tiny)) * (alpha / (om + tiny))
        rho = rho1
        p = r + beta * (p - om * v)
        v = P.dirac(p, kappa, mu)
        alpha = rho / (_dot(r0, v) + tiny)
        s = r - alpha * v
        t = P.dirac(s, kappa, mu)
        om = _dot(t, s) / (_dot(t, t) + tiny)
        x += alpha * p + om * s
        r = s - om * t
        if k % 4 == 3 and bool((_dot(r, r).real <= tol * tol * n0).all()):
            break
    return x


def _solution(dims, U, b, kappa, mu):
    """x = D^-1 b to a 1e-13 residual: complex64 inner solves, complex128 residuals."""
    P, p = _Plain(dims, U, torch.complex128), _Plain(dims, U, torch.complex64)
    b = P.field(b)
    x = torch.zeros_like(b)
    nb = _dot(b, b).real.sqrt()
    for _ in range(20):
        r = b - P.dirac(x, kappa, mu)
        nr = _dot(r, r).real.sqrt()
        if bool((nr <= 1e-13 * nb).all()):
            return x
        nr = torch.where(nr > 0, nr, torch.ones_like(nr))
        x += _inner(p, (r / nr).to(torch.complex64), kappa, mu).to(torch.complex128) * nr
    return None


def _parity(dims):
    x = [torch.arange(n, device="cuda") for n in dims]
    return ((x[3][:, None, None, None] + x[2][None, :, None, None] + x[1][None, None, :, None]
             + x[0][None, None, None, :]) % 2).reshape(-1)


def _network(P, W, r):
    f = P.field(r.reshape(r.shape + (1,)).transpose(-1, -2).flatten(-2))   # spin index c * 4 + s
    off = 0
    for cin, cout in zip(CHANNELS, CHANNELS[1:]):
        w = W[off:off + cout * cin * 144].reshape(cout, cin, 9, 4, 4)
        off += cout * cin * 144
        out = 0
        for k in range(9):
            t = f if k == 0 else P.transport(f, (k - 1) % 4, k <= 4)
            m = w[:, :, k].permute(0, 2, 1, 3).reshape(cout * 4, cin * 4)
            out = out + t @ m.T
        f = out
    return f


def exact(case, seed):
    kind = case["kind"]
    Us, fs = _inputs(case, seed)
    lat = _lattices(case)
    dims, U, f = lat[0], Us[0], fs[0]
    V = _volume(dims)
    kappa, mu = case["kappa"], case.get("mu", 0.0)
    if kind in ("solve", "krylov", "fgcr"):
        if V > 1 << 20:   # too slow in plain torch
            return None
        x = _solution(dims, U, f, kappa, mu)
        return None if x is None else x.reshape(V, 3, 4)
    if kind == "batch":
        if sum(_volume(d) for d in lat) * case["nrhs"] > 1 << 21:
            return None
        xs = [_solution(d, u, b, kappa, 0.0) for d, u, b in zip(lat, Us, fs)]
        return [None if x is None else x.reshape(b.shape) for x, b in zip(xs, fs)]
    P = _Plain(dims, U, torch.complex128)
    if kind == "apply":
        return P.dirac(P.field(f), kappa, mu, case["dagger"]).reshape(V, 3, 4)
    if kind in ("apply_eo", "dslash_eo"):
        odd = _parity(dims)
        p = case["parity"]
        out_sites = (odd == p).nonzero()[:, 0]
        in_sites = out_sites if kind == "apply_eo" else (odd != p).nonzero()[:, 0]
        full = torch.zeros((V, 3, 4), dtype=torch.complex128, device="cuda")
        full[in_sites] = f
        h = P.hop(P.field(full), case["dagger"])
        if kind == "dslash_eo":
            return h.reshape(V, 3, 4)[out_sites]
        t = 2 * kappa * mu * (-1 if case["dagger"] else 1)
        h = P.hop(P.twist(h, -t) / (1 + t * t), case["dagger"])
        return (P.twist(P.field(full), t) - kappa * kappa * h).reshape(V, 3, 4)[out_sites]
    W = _weights(case, seed)
    if kind == "net":
        return _network(P, W, f).reshape(V, 3, 4)
    if V * case["samples"] > 1 << 17:   # too much memory for the graph of operations
        return None
    W = W.requires_grad_(True)
    loss = 0
    for e in f:
        with torch.no_grad():
            r = P.dirac(P.field(e), kappa).reshape(V, 3, 4)
        d = _network(P, W, r).reshape(V, 3, 4) - e
        loss = loss + d.abs().square().sum() / e.abs().square().sum()
    loss.backward()
    return {"loss": float(loss), "grad": W.grad}
