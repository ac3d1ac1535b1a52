"""The measured workloads of the library: whole contour-integral passes on device-resident plans, one-shot
requests, a served mix in shared launches, eigenpairs with polish and left vectors, NLEIGS, Interpol, and two
step entry points, over the sizes of the named workloads (``synth.CONFIGS``) and of the request stream.

The operator is part of the case, as it is of a program that solves one problem again and again; the seed draws
the probe blocks, the start vectors and the steps' dense inputs. (Other operator data would put another number of
eigenvalues inside the region.)

Outputs are eigenvalues, unit eigenvectors and Hankel singular values (or a step's whole result). Residual norms
are left out: they are rounding noise. ``exact`` computes the same quantities in 64 bits with torch and numpy
alone: block elimination of T(z) at the nodes, moments, Hankel SVD, then inverse iteration on each eigenpair.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import synth
from paper_1910_11712_gb300 import binding as nep

FP64, MIXED = nep.NEP_PREC_FP64, nep.NEP_PREC_MIXED


# ------------------------------------------------------------------ the cases
def _pass(name, family, s, N, L, M, precision="mixed", shift=0.0, call="plan"):
    return {"name": name, "call": call, "family": family, "s": s, "N": N, "L": L, "M": M, "precision": precision,
            "shift": shift}


def listed():
    return [
        # the smallest problem a user starts from: 1-D delay equation, every stage bound by latency and launches
        _pass("delay1d_n64_fp64", "delay1d", 64, 32, 16, 4, "fp64"),
        # a small request from host buffers in one call, odd grid: create, solve and read back
        _pass("oneshot_sqrt_s7", "sqrt", 7, 32, 8, 4, call="oneshot"),
        # the headline workload on a plan that the program keeps
        _pass("plan_delay_s64", "delay", 64, 64, 16, 8),
        # the same in plain FP64, for users who do not want complex64 factors
        _pass("plan_delay_s64_fp64", "delay", 64, 64, 16, 8, "fp64"),
        # rational (Drude) problem of bandwidth 128: the widest block of right-hand sides and the most nodes
        _pass("plan_drude_s128", "drude", 128, 128, 32, 8),
        # 3-D square-root problem of bandwidth 576: the widest band
        _pass("plan_sqrt_s24", "sqrt", 24, 64, 24, 8),
        # a ragged mid-size request from host buffers: odd grid, bandwidth above 64
        _pass("oneshot_drude_s97", "drude", 97, 64, 32, 8, shift=-0.25, call="oneshot"),
        # eigenpairs to full accuracy with their left eigenvectors, as resolvent and sensitivity studies want them
        _pass("pairs_delay_s64", "delay", 64, 64, 16, 8, call="pairs"),
        # the rational Krylov solver on the headline problem: one factorisation, many single-vector solves
        {"name": "nleigs_delay_s64", "call": "nleigs", "family": "delay", "s": 64, "krylov": 100, "shift": 0.0,
         "radius": 2.5},
        # a served mix: requests of uneven n, bandwidth, N and L in shared launches
        {"name": "batch_mix6", "call": "batch", "count": 6, "mix": 0, "s_max": 96},
        # the FP64 split-form residual as its own step, the sparse product of every refinement in plain FP64
        {"name": "residual_drude_s128", "call": "residual", "family": "drude", "s": 128, "N": 64, "L": 32, "shift": 0.0},
        # the FP64 moment accumulation as its own step
        {"name": "moments_n16384", "call": "moments", "n": 16384, "N": 64, "L": 32, "K": 16},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["plan", "plan", "plan", "plan", "oneshot", "oneshot", "pairs", "nleigs", "batch", "residual",
                       "moments"])
    shift = round(rng.uniform(-0.5, 0.5), 4)
    if call in ("plan", "oneshot"):
        family = rng.choice(["delay", "delay", "drude", "drude", "sqrt"])
        fp64 = rng.random() < 0.25
        if family == "delay":
            s, L = _log_int(rng, 24, 64 if fp64 else 128), rng.choice([16, 32])
        elif family == "drude":
            s, L = _log_int(rng, 16, 48 if fp64 else 128), rng.choice([8, 16, 32])
        else:
            s, L, shift = _log_int(rng, 6, 12 if fp64 else 20), rng.choice([8, 16, 24]), 0.0
        N = rng.choice([32, 64] if family == "sqrt" else [64, 128])
        return {"call": call, "family": family, "s": s, "N": N, "L": L, "M": 8,
                "precision": "fp64" if fp64 else "mixed", "shift": shift}
    if call == "pairs":
        return {"call": call, "family": "delay", "s": _log_int(rng, 24, 100), "N": rng.choice([64, 128]), "L": 16, "M": 8,
                "precision": "mixed", "shift": shift}
    if call == "nleigs":
        return {"call": call, "family": "delay", "s": _log_int(rng, 24, 80), "krylov": 100, "shift": 0.0,
                "radius": round(rng.uniform(1.0, 2.5), 3)}
    if call == "batch":
        return {"call": call, "count": rng.choice([3, 4, 5, 6]), "mix": rng.randrange(1000), "s_max": 96}
    if call == "residual":
        return {"call": call, "family": rng.choice(["delay", "drude"]), "s": _log_int(rng, 16, 128),
                "N": rng.choice([32, 64]), "L": rng.choice([8, 16, 24, 32]), "shift": shift}
    return {"call": call, "n": _log_int(rng, 256, 16384), "N": rng.choice([32, 64]), "L": rng.choice([8, 16, 24, 32]),
            "K": rng.choice([8, 16])}


# ------------------------------------------------------------------ problems
def _problem(family, s, shift=0.0, radius=None, seed=0):
    """shift 0 is the named workload's own region. Off it, a delay problem takes an ellipse about the dominant real
    eigenvalues: the circle of radius 3 reaches where e^{-z} exceeds 100, and on small grids the diagonal of B alone
    then puts more eigenvalues inside than L * M columns can hold."""
    if family == "delay1d":
        p = synth.delay_1d(n=s, seed=seed)
        p.region = {"center": -0.9 + 0j, "a": 0.9, "b": 0.45}
        return p
    if family == "delay":
        p = synth.delay_2d(s=s, seed=seed)
        if shift:
            p.region = {"center": complex(-1.5 + shift), "a": 1.5, "b": 0.75}
        elif radius:
            p.region = {"center": -2.0 + 0j, "a": radius, "b": radius}
        return p
    if family == "drude":
        return synth.drude_2d(s=s, seed=seed, center=2.0 + shift)
    return synth.sqrt_3d(s=s, seed=seed)


def _requests(case):
    """The problems of a served mix, from the request stream's own draw."""
    out = []
    for r in synth.serving_requests(case["count"], seed=case["mix"], s_max=case["s_max"]):
        family = r["family"]
        s, L = (r["s"], r["L"]) if family == "drude" else (max(24, r["s"]), max(16, r["L"]))
        out.append((_problem(family, s, r["shift"], seed=r["seed"]), max(64, r["N"]), L, 8))
    return out


def _probe(n, L, seed):
    return synth.random_probe_block(n, L, seed)


def _on_device(a):
    a = np.asarray(a)
    return torch.from_numpy(np.ascontiguousarray(a.ravel(order="F")).view(np.float64).copy()).cuda()


def _randn(count, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(count, dtype=torch.float64, device="cuda", generator=g)


def _precision(case):
    return FP64 if case["precision"] == "fp64" else MIXED


# ------------------------------------------------------------------ prepare
def prepare(case, seed):
    call = case["call"]
    if call == "moments":
        n, N, L, K = case["n"], case["N"], case["L"], case["K"]
        j = np.arange(N)
        zeta = np.exp(2j * np.pi * (j + 0.5) / N)
        coef = (zeta[None, :] / N * zeta[None, :] ** np.arange(K)[:, None]) * (1.0 + (seed % 7) / 16)
        return {"call": call, "n": n, "N": N, "L": L, "K": K,
                "coef": torch.from_numpy(coef.reshape(-1).view(np.float64).copy()).cuda(),
                "Y": _randn(N * n * L * 2, seed),
                "S": torch.empty(K * n * L * 2, dtype=torch.float64, device="cuda")}
    if call == "batch":
        reqs = _requests(case)
        splits = [nep.Split.from_problem(p) for p, _, _, _ in reqs]
        plans = [nep.Plan(sp, p.region, N, L, M, precision=MIXED) for sp, (p, N, L, M) in zip(splits, reqs)]
        return {"call": call, "splits": splits, "plans": plans,
                "V": [_on_device(_probe(p.n, L, seed + k)) for k, (p, _, L, _) in enumerate(reqs)]}
    p = _problem(case["family"], case["s"], case["shift"], case.get("radius"))
    split = nep.Split.from_problem(p)
    state = {"call": call, "case": case, "region": p.region, "split": split}
    if call == "residual":
        N, L = case["N"], case["L"]
        z, _, _ = nep.nodes(p.region, N)
        F, _ = nep.coefficients(split, z)
        state.update(F=_on_device(F), V=_on_device(_probe(p.n, L, seed)), Y=_randn(N * p.n * L * 2, seed),
                     R=torch.empty(N * p.n * L * 2, dtype=torch.float64, device="cuda"))
    elif call == "oneshot":
        state["V"] = _probe(p.n, case["L"], seed)
    elif call in ("plan", "pairs"):
        state["V"] = _on_device(_probe(p.n, case["L"], seed))
        state["plan"] = nep.Plan(split, p.region, case["N"], case["L"], case["M"], precision=_precision(case))
        if call == "pairs":
            state["Y"] = torch.empty(p.n * 64 * 2, dtype=torch.float64, device="cuda")
            state["eta"] = torch.empty(64, dtype=torch.float64, device="cuda")
    else:
        state["seed"] = seed
    return state


# ------------------------------------------------------------------ run
def _order(lam):
    """By real part, then imaginary part; the real parts of a conjugate pair agree to rounding only."""
    return np.lexsort((lam.imag, np.round(lam.real, 8)))


def _eigenpairs(res):
    at = _order(res["lam"])
    return {"lam": res["lam"][at], "X": res["X"][:, at], "sigma": res["sigma"]}


def run(state):
    call = state["call"]
    if call == "plan":
        state["plan"].execute(state["V"])
        return _eigenpairs(state["plan"].result())
    if call == "oneshot":
        c = state["case"]
        return _eigenpairs(nep.ciss_solve(state["split"], state["region"], c["N"], c["L"], c["M"], state["V"],
                                          precision=_precision(c)))
    if call == "batch":
        nep.execute_batch(state["plans"], state["V"])
        return [_eigenpairs(p.result()) for p in state["plans"]]
    if call == "pairs":
        plan = state["plan"]
        plan.execute(state["V"])
        plan.polish(tol=1e-13)
        k, _ = plan.left(state["Y"], state["eta"], 64)
        res = plan.result()
        at, n = _order(res["lam"]), state["split"].n
        Y = torch.view_as_complex(state["Y"][:k * n * 2].view(k, n, 2))
        return {"lam": res["lam"][at], "X": res["X"][:, at], "Y": Y[torch.from_numpy(at).cuda()].T}
    if call == "nleigs":
        res = nep.nleigs_solve(state["split"], state["region"], krylov=state["case"]["krylov"], seed=state["seed"])
        at = _order(res["lam"])
        return {"lam": res["lam"][at], "X": res["X"][:, at]}
    if call == "residual":
        c = state["case"]
        nep.split_residual(state["split"], c["N"], state["F"], c["L"], state["V"], state["Y"], state["R"])
        return state["R"]
    nep.moments(state["n"], state["L"], state["N"], state["K"], state["coef"], state["Y"], state["S"])
    return state["S"]


# ------------------------------------------------------------------ work
def _pass_work(p, N, L, M):
    """Least work of a pass: band LU and one solve per node, the moments; operator and V in, eigenpairs out."""
    n = p.n
    kl = p.meta["bandwidth"]
    nnz = sum(A.nnz for A in p.mats)
    flops = N * (8.0 * n * kl * 2 * kl + 8.0 * n * 3 * kl * L) + 8.0 * 2 * M * n * L * N
    return {"bytes": 16.0 * n * L + 12.0 * nnz + 16.0 * n * 10 + 8.0 * L * M, "flops": flops}


def work(case):
    call = case["call"]
    if call == "moments":
        c = 1.0 * case["n"] * case["L"]
        return {"bytes": 16.0 * c * (case["N"] + case["K"]), "flops": 8.0 * c * case["N"] * case["K"]}
    if call == "batch":
        parts = [_pass_work(*r) for r in _requests(case)]
        return {k: sum(w[k] for w in parts) for k in ("bytes", "flops")}
    p = _problem(case["family"], case["s"], case["shift"])
    if call == "residual":
        N, L, c = case["N"], case["L"], 1.0 * p.n * case["L"]
        nnz = sum(A.nnz for A in p.mats)
        return {"bytes": 16.0 * c * (2 * N + 1) + 12.0 * nnz, "flops": 8.0 * p.mats[0].nnz * L * N}
    if call == "nleigs":
        kl, d = p.meta["bandwidth"], 27  # one band LU, one solve per Arnoldi step, two Gram-Schmidt passes on d n-vectors
        k = case["krylov"]
        return {"bytes": 16.0 * p.n * 10 + 12.0 * sum(A.nnz for A in p.mats),
                "flops": 8.0 * p.n * kl * 2 * kl + k * 8.0 * p.n * 3 * kl + 8.0 * 2 * p.n * k * (k + d)}
    w = _pass_work(p, case["N"], case["L"], case["M"])
    if call == "pairs":
        kl = p.meta["bandwidth"]
        w["flops"] += 2 * 8 * 8.0 * p.n * kl * 2 * kl
        w["bytes"] += 16.0 * p.n * 10
    return w


# ------------------------------------------------------------------ exact
def _fn(spec, z):
    """f(z) and f'(z) of one function description."""
    al, be = complex(spec.get("alpha", 1)), complex(spec.get("beta", 1))
    x = al * np.asarray(z, np.complex128)
    if spec["kind"] == "exp":
        return be * np.exp(x), be * al * np.exp(x)
    if spec["kind"] == "sqrt":
        r = np.sqrt(x - complex(spec["shift"]))
        return be * r, be * al * 0.5 / r
    num, den = np.array(spec["num"]), np.array(spec["den"] if spec["den"] is not None else [1.0])
    p, q = np.polyval(num, x), np.polyval(den, x)
    dp, dq = np.polyval(np.polyder(num), x), np.polyval(np.polyder(den), x)
    return be * p / q, be * al * (dp * q - p * dq) / (q * q)


class _Blocks:
    """T(z) at several z as a block tridiagonal matrix whose off-diagonal blocks are diagonal."""

    def __init__(self, p, z, dev):
        b = p.meta.get("grid", p.n) if p.name != "sqrt_3d" else p.meta["grid"] ** 2
        self.b, self.K, self.dev = b, p.n // b, dev
        f, df = zip(*(_fn(s, z) for s in p.fns))
        self.f, self.df = (torch.from_numpy(np.array(v)).to(dev) for v in (f, df))  # terms x points
        self.diag, self.lo, self.up = [], [], []
        for A in p.mats:
            A = A.tocoo()
            D = torch.zeros(self.K, b, b, dtype=torch.float64)
            same = A.row // b == A.col // b
            D[A.row[same] // b, A.row[same] % b, A.col[same] % b] = torch.from_numpy(A.data[same])
            off = [torch.zeros(p.n, dtype=torch.float64) for _ in range(2)]
            for o, sign in zip(off, (-1, 1)):
                at = A.col - A.row == sign * b
                o[A.row[at]] = torch.from_numpy(A.data[at])
            if self.K > 1 and np.any(~same & (np.abs(A.col - A.row) != b)):
                raise ValueError("not block tridiagonal")
            self.diag.append(D.to(dev))
            self.lo.append(off[0].to(dev))
            self.up.append(off[1].to(dev))

    def block(self, k, f=None):
        f = self.f if f is None else f
        return sum(fi[:, None, None] * D[k] for fi, D in zip(f, self.diag))

    def couple(self, side, k, f=None):
        f = self.f if f is None else f
        rows = slice(k * self.b, (k + 1) * self.b)
        return sum(fi[:, None] * o[rows] for fi, o in zip(f, side))[:, :, None]

    def factor(self):
        self.inv = []
        for k in range(self.K):
            D = self.block(k)
            if k:
                D = D - self.couple(self.lo, k) * self.inv[-1] * self.couple(self.up, k - 1).transpose(1, 2)
            self.inv.append(torch.linalg.inv(D))

    def apply(self, x, f=None):
        b, out = self.b, torch.empty_like(x)
        for k in range(self.K):
            r = self.block(k, f) @ x[:, k * b:(k + 1) * b]
            if k:
                r = r + self.couple(self.lo, k, f) * x[:, (k - 1) * b:k * b]
            if k + 1 < self.K:
                r = r + self.couple(self.up, k, f) * x[:, (k + 1) * b:(k + 2) * b]
            out[:, k * b:(k + 1) * b] = r
        return out

    def solve(self, r):
        b, y = self.b, r.clone()
        for k in range(1, self.K):
            y[:, k * b:(k + 1) * b] -= self.couple(self.lo, k) * (self.inv[k - 1] @ y[:, (k - 1) * b:k * b])
        for k in range(self.K - 1, -1, -1):
            t = y[:, k * b:(k + 1) * b]
            if k + 1 < self.K:
                t = t - self.couple(self.up, k) * y[:, (k + 1) * b:(k + 2) * b]
            y[:, k * b:(k + 1) * b] = self.inv[k] @ t
        return y


def _unit(x):
    """Unit 2-norm columns, first entry of largest modulus real positive."""
    x = x / np.linalg.norm(x, axis=0)
    big = np.take_along_axis(x, np.abs(x).argmax(axis=0)[None, :], 0)
    return x * (np.abs(big) / big)


def _exact_pass(p, N, L, M, V, dev):
    """Eigenpairs inside the region and the Hankel singular values, in 64 bits."""
    c, a, b = p.region["center"], p.region["a"], p.region["b"]
    th = 2 * np.pi * (np.arange(N) + 0.5) / N
    z = c + a * np.cos(th) + 1j * b * np.sin(th)
    w, zeta = (b * np.cos(th) + 1j * a * np.sin(th)) / N, (z - c) / a
    T = _Blocks(p, z, dev)
    T.factor()
    Vd = torch.from_numpy(V).to(dev)
    B = Vd.expand(N, -1, -1)
    Y = T.solve(B)
    for _ in range(2):
        Y = Y + T.solve(B - T.apply(Y))
    T.inv = None
    C = torch.from_numpy(w[None, :] * zeta[None, :] ** np.arange(2 * M)[:, None]).to(dev)
    S = torch.einsum("kj,jnl->knl", C, Y)
    mu = torch.einsum("nl,knm->klm", Vd.conj(), S).cpu().numpy()
    H = np.block([[mu[i + j] for j in range(M)] for i in range(M)])
    H1 = np.block([[mu[i + j + 1] for j in range(M)] for i in range(M)])
    U, sig, Wh = np.linalg.svd(H)
    m = int((sig > 1e-12 * sig[0]).sum())
    W = Wh[:m].conj().T / sig[:m]
    th1, Q = np.linalg.eig(U[:, :m].conj().T @ H1 @ W)
    lam = c + a * th1
    S0 = S[:M].permute(1, 0, 2).reshape(p.n, M * L).cpu().numpy()
    X = S0 @ (W @ Q)
    near = ((lam - c).real / a) ** 2 + ((lam - c).imag / b) ** 2 < 1.02
    return _exact_pairs(p, lam[near], X[:, near], dev) + (sig,)


def _exact_pairs(p, lam, X, dev):
    """Inverse iteration from estimates; the distinct pairs strictly inside the region, sorted by (Re, Im)."""
    c, a, b = p.region["center"], p.region["a"], p.region["b"]
    x = torch.from_numpy(np.ascontiguousarray((X / np.linalg.norm(X, axis=0)).T)).to(dev)[:, :, None]
    for it in range(6):
        T = _Blocks(p, lam, dev)
        T.factor()
        y = T.solve(T.apply(x, T.df))
        step = (x[:, :, 0].conj() * y[:, :, 0]).sum(1).cpu().numpy()
        x = y / torch.linalg.norm(y, dim=1, keepdim=True)
        lam = lam - np.where(np.isfinite(step) & (step != 0), 1 / step, 0)
    T = _Blocks(p, lam, dev)
    r = torch.linalg.norm(T.apply(x)[:, :, 0], dim=1).cpu().numpy()
    norms = np.array([abs(A).sum(axis=1).max() for A in p.mats])
    scale = (T.f.abs().cpu().numpy() * norms[:, None]).sum(0)
    ok = ((lam - c).real / a) ** 2 + ((lam - c).imag / b) ** 2 < 1
    ok &= r <= 1e-11 * scale
    keep = []
    for i in np.flatnonzero(ok):
        if all(abs(lam[i] - lam[j]) > 1e-9 * max(1, abs(lam[i])) for j in keep):
            keep.append(int(i))
    keep = np.array(keep, dtype=int)
    keep = keep[_order(lam[keep])]
    return lam[keep], np.asfortranarray(_unit(x[keep, :, 0].cpu().numpy().T))


def _exact_left(p, lam, X):
    """Left vectors of a complex symmetric T: y = conj(x) up to the scaling y^* T'(lam) x = 1."""
    Y = np.conj(X)
    for i, l in enumerate(lam):
        d = sum(_fn(s, l)[1] * (A @ X[:, i]) for s, A in zip(p.fns, p.mats))
        Y[:, i] /= np.conj(X[:, i] @ d)
    return Y


def exact(case, seed):
    call = case["call"]
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if call == "moments":
        st = prepare(case, seed)
        Y = torch.view_as_complex(st["Y"].view(st["N"], -1, 2))
        return torch.view_as_real(torch.view_as_complex(st["coef"].view(st["K"], st["N"], 2)) @ Y).reshape(-1)
    if call == "batch":
        out = []
        for k, (p, N, L, M) in enumerate(_requests(case)):
            lam, X, sig = _exact_pass(p, N, L, M, _probe(p.n, L, seed + k), dev)
            out.append({"lam": lam, "X": X, "sigma": sig})
        return out
    p = _problem(case["family"], case["s"], case["shift"], case.get("radius"))
    if call == "residual":
        N, L, n = case["N"], case["L"], p.n
        Y = torch.view_as_complex(_randn(N * n * L * 2, seed).view(N, L, n, 2))
        th = 2 * np.pi * (np.arange(N) + 0.5) / N
        z = p.region["center"] + p.region["a"] * np.cos(th) + 1j * p.region["b"] * np.sin(th)
        R = torch.from_numpy(np.ascontiguousarray(_probe(n, L, seed).T)).to(dev).repeat(N, 1, 1)
        for s, A in zip(p.fns, p.mats):
            f, A = torch.from_numpy(_fn(s, z)[0]).to(dev)[:, None, None], A.tocoo()
            for o in np.unique(A.col - A.row):
                at = A.col - A.row == o
                v = torch.zeros(n, dtype=torch.float64)
                v[A.row[at]] = torch.from_numpy(A.data[at])
                r0, r1 = max(0, -o), n - max(0, o)
                R[:, :, r0:r1] -= f * v[r0:r1].to(dev) * Y[:, :, r0 + o:r1 + o]
        return torch.view_as_real(R).reshape(-1)
    if call == "nleigs":
        lam, X, _ = _exact_pass(p, 64, 16, 8, _probe(p.n, 16, seed), dev)
        return {"lam": lam, "X": X}
    lam, X, sig = _exact_pass(p, case["N"], case["L"], case["M"], _probe(p.n, case["L"], seed), dev)
    if call == "pairs":
        return {"lam": lam, "X": X, "Y": _exact_left(p, lam, X)}
    return {"lam": lam, "X": X, "sigma": sig}
