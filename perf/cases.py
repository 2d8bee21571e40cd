"""Timed cases of the eigensolver: whole solves, batches and gradients, and the steps of one outer iteration.

Every case goes through the package's public wrapper (`Chase`, `ChaseEigh`).  Matrices are A = Q diag(lam) Q^H with Q
a product of eight seeded Householder reflectors, generated on the GPU, so exact eigenpairs are known without an
eigensolve.  Matrix arguments are column-major storages, as the wrapper takes them: a (cols x rows) tensor per
rows x cols matrix.  Eigenvectors are defined up to a phase; each is returned with the phase that makes its inner
product with the first start vector real and positive, which is what a program that keeps or compares them does too.
"""
import math
import random

import torch

from paper_2205_02491_gb300 import Chase, ChaseEigh

DEV = "cuda:0"
REFLECTORS = 8
RUNS, STEPS = 4, 25  # Lanczos runs and steps (the library's defaults)


def listed():
    return [
        # the smallest problem: launches and latency count
        dict(name="solve_c512", kind="solve", n=512, nev=16, nex=8, cplx=True, mode="fp64", spectrum="unit"),
        # a real dense problem in the shape of the eigen-type suite (nev 7.5 %, nex 2.5 %), geometric spectrum
        dict(name="solve_r2000", kind="solve", n=2000, nev=150, nex=50, cplx=False, mode="fp64", spectrum="geometric"),
        # the mixed-precision solve: split-BF16 bulk sweeps, then FP64 sweeps
        dict(name="solve_c3001_mixed", kind="solve", n=3001, nev=150, nex=75, cplx=True, mode="bf16x6", spectrum="unit"),
        # many problems of uneven size in one call (a set of independent k-points)
        dict(name="batch_c512_2048", kind="batch", nprob=8, nmin=512, nmax=2048, sizes=4, cplx=True, mode="fp64", spectrum="unit"),
        # the filter of a first outer iteration: every column at the initial degree
        dict(name="filter_c8192", kind="filter", n=8192, k=437, cplx=True, mode="fp64", spectrum="low", degmin=20, degmax=20),
        # the largest block: a late iteration, each column at its own degree
        dict(name="filter_c20000", kind="filter", n=20000, k=800, cplx=True, mode="fp64", spectrum="low", degmin=2, degmax=7),
        # the bulk filter of a mixed-precision solve, odd sizes, real
        dict(name="filter_r5003_mixed", kind="filter", n=5003, k=333, cplx=False, mode="bf16x3", spectrum="low", degmin=4, degmax=20),
        # orthonormalisation of a filtered block against locked vectors
        dict(name="qr_c8192", kind="qr", n=8192, k=437, locked=120, cplx=True),
        # Rayleigh-Ritz of a filtered block (projection, small eigensolve, back-transform, residuals)
        dict(name="rr_c8192", kind="rr", n=8192, k=437, cplx=True, spectrum="low"),
        # the same, real, odd and ragged
        dict(name="rr_r6001", kind="rr", n=6001, k=291, cplx=False, spectrum="low"),
        # spectral bounds before the first filter
        dict(name="lanczos_c8192", kind="lanczos", n=8192, k=437, cplx=True, spectrum="low"),
        # forward and backward of an eigenvalue/eigenvector loss (a training step through the eigensolver)
        dict(name="grad_r4096", kind="grad", n=4096, nev=64, nex=32, cplx=False, mode="fp64", spectrum="unit"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "batch", "filter", "filter", "filter", "qr", "rr", "rr", "lanczos", "grad"])
    cplx = rng.random() < 0.6
    if kind == "solve":
        n = _log_int(rng, 300, 3000)
        nev = max(8, int(n * rng.uniform(0.02, 0.075)))
        return dict(kind=kind, n=n, nev=nev, nex=max(4, nev // rng.choice([2, 3])), cplx=cplx,
                    mode=rng.choice(["fp64", "fp64", "bf16x6", "bf16x3"]), spectrum=rng.choice(["unit", "low", "geometric"]))
    if kind == "batch":
        nmin = _log_int(rng, 300, 700)
        return dict(kind=kind, nprob=rng.randint(3, 8), nmin=nmin, nmax=_log_int(rng, nmin + 100, 2000),
                    sizes=rng.randrange(1 << 20), cplx=True, mode="fp64", spectrum="unit")
    if kind == "grad":
        nev = rng.randint(8, 64)
        return dict(kind=kind, n=_log_int(rng, 700, 4096), nev=nev, nex=max(4, nev // 2), cplx=False, mode="fp64",
                    spectrum="unit")
    n = _log_int(rng, 500, 12000)
    if kind == "lanczos":
        return dict(kind=kind, n=n, k=max(8, n // rng.randint(15, 40)), cplx=cplx, spectrum="low")
    k = _log_int(rng, 8, max(24, n // 15))
    if kind == "filter":
        lo = rng.randint(1, 12)
        return dict(kind=kind, n=n, k=k, cplx=cplx, mode=rng.choice(["fp64", "fp64", "bf16x6", "bf16x3"]),
                    spectrum="low", degmin=lo, degmax=rng.randint(lo, 20))
    if kind == "qr":
        return dict(kind=kind, n=n, k=k, locked=rng.choice([0, k // 3, (2 * k) // 3]), cplx=cplx)
    return dict(kind=kind, n=n, k=k, cplx=cplx, spectrum="low")


# ------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _dtype(cplx):
    return torch.complex128 if cplx else torch.float64


def _normal(g, shape, cplx):
    return torch.randn(shape, generator=g, device=DEV, dtype=_dtype(cplx))


def _stratified(g, count, lo, hi):
    """`count` ascending values on [lo, hi], uniform within cells of equal width, gaps of at least half a cell."""
    u = torch.rand(count, generator=g, device=DEV, dtype=torch.float64)
    return lo + (hi - lo) / count * (torch.arange(count, device=DEV, dtype=torch.float64) + 0.5 * u)


def _spectrum(g, kind, n):
    if kind == "unit":
        return _stratified(g, n, -1.0, 1.0)
    if kind == "low":  # the wanted end on [-2, 0], the rest up to 50
        nlow = max(2, n // 8)
        return torch.cat([_stratified(g, nlow, -2.0, 0.0), _stratified(g, n - nlow, 0.0, 50.0)])
    # geometric law on [-1, -1e-4], sparse at the wanted end; jittered within a quarter of the ratio between neighbours
    x = torch.arange(n, device=DEV, dtype=torch.float64) + 0.25 * torch.rand(n, generator=g, device=DEV, dtype=torch.float64)
    return -torch.pow(torch.tensor(1e-4, device=DEV, dtype=torch.float64), x / n)


def _storage_of(lam, U):
    """Column-major storage of A = Q diag(lam) Q^H, Q = H_1 ... H_r with the reflectors' vectors in U's rows."""
    S = torch.diag(lam.to(U.dtype))
    for u in reversed(U.conj()):  # the storage is A^T = conj(A)
        tau = (2.0 / (u.abs().square().sum())).item()
        S.addr_(u, (u.conj() @ S), alpha=-tau)
        S.addr_((S @ u), u.conj(), alpha=-tau)
    n = S.shape[0]
    for i in range(0, n, 2048):  # exactly Hermitian, block by block
        for j in range(0, i + 1, 2048):
            m = 0.5 * (S[i:i + 2048, j:j + 2048] + S[j:j + 2048, i:i + 2048].mH)
            S[i:i + 2048, j:j + 2048] = m
            S[j:j + 2048, i:i + 2048] = m.mH
    return S


def _eigvec_storage(U, count):
    """Rows Q e_i, i < count: the storage of the exact eigenvectors of the lowest `count` eigenvalues."""
    E = torch.zeros((count, U.shape[1]), dtype=U.dtype, device=DEV)
    E[torch.arange(count), torch.arange(count)] = 1.0
    for u in reversed(U):
        tau = 2.0 / u.abs().square().sum()
        E.addr_(E @ u.conj(), u, alpha=-tau.item())
    return E


def _fix_phase(Vt, ref):
    c = Vt @ ref.conj()
    return Vt * (c.conj() / c.abs())[:, None]


def _sizes(case):
    r = random.Random(case["sizes"])
    ns = [r.randint(case["nmin"], case["nmax"]) for _ in range(case["nprob"])]
    return [(n, max(1, round(0.05 * n)), max(1, round(0.05 * n) // 2)) for n in ns]


def _problem(g, n, m, cplx, spectrum):
    """lam, reflector vectors, an n x m start block and the Lanczos start vectors (as storages)."""
    lam = _spectrum(g, spectrum, n)
    U = _normal(g, (REFLECTORS, n), cplx)
    return lam, U, _normal(g, (m, n), cplx), _normal(g, (RUNS, n), cplx)


def _degrees(case):
    r = random.Random(case["k"])
    return sorted(r.randint(case["degmin"], case["degmax"]) for _ in range(case["k"]))


def _filter_bounds(lam, k):
    """(b_sup, mu_1, mu_ne) as the bounds of a block of k columns stand."""
    return float(lam[-1]) * 1.001, float(lam[0]), float(lam[k])


def _inputs(case, seed):
    """The case's inputs, made from the seed alone (without the library)."""
    g = _gen(seed)
    kind, cplx = case["kind"], case["cplx"]
    if kind in ("solve", "grad"):
        d = dict(zip(("lam", "U", "V0", "L0"), _problem(g, case["n"], case["nev"] + case["nex"], cplx, case["spectrum"])))
        if kind == "grad":
            d["weights"] = torch.randn(case["nev"], generator=g, device=DEV, dtype=torch.float64)
            B = torch.randn((case["n"], case["n"]), generator=g, device=DEV, dtype=torch.float64)
            d["B"] = 0.5 * (B + B.mT)
        return d
    if kind == "batch":
        return dict(problems=[_problem(g, n, nev + nex, cplx, case["spectrum"]) for n, nev, nex in _sizes(case)])
    n, k = case["n"], case["k"]
    if kind == "qr":
        # locked orthonormal columns, then a block whose directions were amplified unevenly (condition about 1e4)
        l = case["locked"]
        m = k - l
        Y = _eigvec_storage(_normal(g, (REFLECTORS, n), cplx), l)
        P = torch.linalg.qr(_normal(g, (m, m), cplx))[0]
        scale = torch.logspace(0, -4, m, device=DEV, dtype=torch.float64)
        X = (P * scale[None, :]) @ _normal(g, (m, n), cplx)
        return dict(X=torch.cat([Y, X]))
    lam, U, V0, L0 = _problem(g, n, k, cplx, case["spectrum"])
    d = dict(lam=lam, U=U, V0=V0, L0=L0)
    if kind == "rr":
        # an orthonormal block near the lowest eigenvectors, mixed, as the filter and QR leave it
        E = _eigvec_storage(U, k)
        P = torch.linalg.qr(_normal(g, (k, k), cplx))[0]
        d["Q"] = torch.linalg.qr((P @ E + 1e-4 * V0).mT)[0].mT.contiguous()
    return d


def prepare(case, seed):
    d = _inputs(case, seed)
    kind, cplx = case["kind"], case["cplx"]
    s = dict(case=dict(case), **{k: d[k] for k in ("V0", "L0", "Q", "X", "weights", "B") if k in d})
    if kind == "batch":
        s["dims"] = _sizes(case)
        s["A"] = [_storage_of(lam, U) for lam, U, _, _ in d["problems"]]
        s["V0"] = [p[2] for p in d["problems"]]
        s["L0"] = [p[3] for p in d["problems"]]
        s["solver"] = Chase(max(x[0] for x in s["dims"]), max(x[1] + x[2] for x in s["dims"]), complex_=cplx,
                            opts=dict(batch_workers=8))
        return s
    if kind != "qr":
        s["A"] = _storage_of(d["lam"], d["U"])
    if kind in ("solve", "grad"):
        s["solver"] = Chase(case["n"], case["nev"] + case["nex"], complex_=cplx)
    else:
        s["solver"] = Chase(case["n"], case["k"], complex_=cplx)
    if kind == "filter":
        s["degrees"], s["bounds"] = _degrees(case), _filter_bounds(d["lam"], case["k"])
    return s


def run(s):
    c, solver = s["case"], s["solver"]
    kind = c["kind"]
    if kind == "solve":
        w, Vt = solver.solve(s["A"], c["nev"], c["nex"], 1e-10, 20, c["mode"], s["V0"], s["L0"])
        return w, _fix_phase(Vt, s["V0"][0])
    if kind == "batch":
        V = [v.clone() for v in s["V0"]]  # replaced by the eigenvectors and the next start block
        ws, _ = solver.solve_batched(s["A"], [x[1] for x in s["dims"]], [x[2] for x in s["dims"]], 1e-10, 20, c["mode"],
                                     V, s["L0"])
        return ws, [_fix_phase(v, v0[0]) for v, v0 in zip(V, s["V0"])]
    if kind == "grad":
        A = s["A"].detach().requires_grad_(True)
        w, V = ChaseEigh.apply(A, solver, c["nev"], c["nex"], 1e-10, 20, c["mode"], s["V0"], s["L0"])
        loss = (s["weights"] * w).sum() + (V.mT @ (s["B"] @ V)).square().sum()
        loss.backward()
        return w.detach(), _fix_phase(V.detach().mT, s["V0"][0]), A.grad
    if kind == "filter":
        return solver.filter(s["A"], s["V0"].clone(), s["degrees"], *s["bounds"], mode=c["mode"])
    if kind == "qr":
        return solver.qr(s["X"].clone(), c["locked"])
    if kind == "rr":
        Q = s["Q"].clone()
        w, r = solver.rayleigh_ritz(s["A"], Q)
        return w, r, _fix_phase(Q, s["V0"][0])
    b = solver.lanczos(s["A"], c["k"], s["L0"], RUNS, STEPS)
    return [b["b_sup"], b["mu_1"], b["mu_ne"], b["theta_max"]]


# ------------------------------------------------------------------ what a pass cannot do without
def _solve_work(n, nev, nex, cplx, deg=20):
    e, f, ne = (16, 8, nev + nex) if cplx else (8, 2, nev + nex)
    return e * (n * n + 2 * n * ne), f * n * n * (RUNS * STEPS + (deg + 1) * ne) + 4 * f * n * ne * ne


def work(case):
    kind, cplx = case["kind"], case["cplx"]
    e, f = (16, 8) if cplx else (8, 2)
    if kind == "solve":  # the Lanczos bounds and one outer iteration at the initial degree
        b, fl = _solve_work(case["n"], case["nev"], case["nex"], cplx)
    elif kind == "batch":
        parts = [_solve_work(n, nev, nex, cplx) for n, nev, nex in _sizes(case)]
        b, fl = sum(p[0] for p in parts), sum(p[1] for p in parts)
    elif kind == "grad":  # the solve, and a gradient written from one product with every eigenvector
        b, fl = _solve_work(case["n"], case["nev"], case["nex"], cplx)
        b, fl = b + 16 * case["n"] ** 2, fl + 4 * case["n"] ** 2 * case["nev"]
    else:
        n, k = case["n"], case["k"]
        b = e * (n * n + 2 * n * k)
        if kind == "filter":
            fl = f * n * n * sum(_degrees(case))
        elif kind == "qr":
            b, fl = e * 2 * n * k, 2 * f * n * k * k
        elif kind == "rr":
            fl = f * (n * n * k + 3 * n * k * k + 4 * k ** 3)
        else:
            b, fl = e * (n * n + n * RUNS), f * n * n * RUNS * STEPS
    return {"bytes": b, "flops": fl}


# ------------------------------------------------------------------ the same in plain 64-bit torch
def _exact_filter(A, X, degrees, b_sup, mu_1, mu_ne):
    """A, X: n x n and n x k.  Scaled three-term Chebyshev recurrence; column a takes degrees[a] products."""
    c, e = 0.5 * (b_sup + mu_ne), 0.5 * (b_sup - mu_ne)
    sigma1 = e / (mu_1 - c)
    out = X.clone()
    prev, cur, sigma, first = None, X, sigma1, 0
    for step in range(1, degrees[-1] + 1):
        skip = sum(1 for d in degrees if d < step) - first
        first += skip
        cur = cur[:, skip:]
        prev = None if prev is None else prev[:, skip:]
        if step == 1:
            nxt = (sigma1 / e) * (A @ cur - c * cur)
        else:
            s2 = 1.0 / (2.0 / sigma1 - sigma)
            nxt = (2.0 * s2 / e) * (A @ cur - c * cur) - sigma * s2 * prev
            sigma = s2
        prev, cur = cur, nxt
        done = sum(1 for d in degrees if d == step)
        out[:, first:first + done] = cur[:, :done]
    return out


def _exact_lanczos(A, L0, ne):
    n, thetas, weights, sup = A.shape[0], [], [], []
    for r in range(RUNS):
        Q = [L0[:, r] / torch.linalg.vector_norm(L0[:, r])]
        alpha, beta = [], []
        for j in range(STEPS):
            w = A @ Q[j]
            a = torch.vdot(Q[j], w).real
            w = w - a * Q[j] - (beta[-1] * Q[j - 1] if j else 0.0)
            for _ in range(2):
                M = torch.stack(Q, 1)
                w = w - M @ (M.mH @ w)
            alpha.append(a)
            beta.append(torch.linalg.vector_norm(w))
            Q.append(w / beta[-1])
        off = torch.stack(beta[:-1])
        T = torch.diag(torch.stack(alpha)) + torch.diag(off, 1) + torch.diag(off, -1)
        th, Z = torch.linalg.eigh(T)
        thetas.append(th)
        weights.append(Z[0].square() / RUNS)
        sup.append(th[-1] + beta[-1])
    theta, order = torch.sort(torch.cat(thetas))
    total = torch.cumsum(torch.cat(weights)[order], 0)
    b_sup, mu_1 = max(sup).item(), theta[0].item()
    at = int((total < ne / n).sum())
    span = b_sup - mu_1
    mu_ne = min(max(theta[min(at, len(theta) - 1)].item(), mu_1 + 1e-3 * span), b_sup - 1e-3 * span)
    return [b_sup, mu_1, mu_ne, theta[-1].item()]


def exact(case, seed):
    d = _inputs(case, seed)
    kind = case["kind"]
    if kind == "solve":
        nev = case["nev"]
        return d["lam"][:nev], _fix_phase(_eigvec_storage(d["U"], nev), d["V0"][0])
    if kind == "batch":  # the part of a block behind the wanted pairs is a start block without an exact value
        return [p[0][:x[1]] for p, x in zip(d["problems"], _sizes(case))], [None for _ in d["problems"]]
    if kind == "qr":
        Q, R = torch.linalg.qr(d["X"].mT)
        r = torch.diagonal(R)
        Q = Q * (r / r.abs())[None, :]
        return torch.cat([d["X"][:case["locked"]], Q[:, case["locked"]:].mT])
    if kind == "grad":
        n, nev = case["n"], case["nev"]
        lam, Qt = d["lam"], _eigvec_storage(d["U"], n)
        V = Qt[:nev].mT
        BV = d["B"] @ V
        gV = 4.0 * BV @ (V.mT @ BV)
        gap = lam[None, :nev] - lam[:, None]
        gap[torch.arange(nev), torch.arange(nev)] = math.inf
        inner = (Qt @ gV) / gap
        inner[torch.arange(nev), torch.arange(nev)] = d["weights"]
        G = (Qt.mT @ inner) @ V.mT
        return lam[:nev], _fix_phase(Qt[:nev], d["V0"][0]), 0.5 * (G + G.mT)
    A = _storage_of(d["lam"], d["U"]).mT
    if kind == "filter":
        k = case["k"]
        return _exact_filter(A, d["V0"].mT, _degrees(case), *_filter_bounds(d["lam"], k)).mT.contiguous()
    if kind == "rr":
        Q = d["Q"].mT
        W = A @ Q
        G = Q.mH @ W
        w, Z = torch.linalg.eigh(0.5 * (G + G.mH))
        V = Q @ Z
        res = torch.linalg.vector_norm(W @ Z - V * w[None, :], dim=0)
        return w, res, _fix_phase(V.mT, d["V0"][0])
    return _exact_lanczos(A, d["L0"].mT, case["k"])
