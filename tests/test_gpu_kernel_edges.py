"""Kernels at the sizes where their tiles, clusters and dispatch lines end: Lanczos products and Ritz values, small
Hermitian eigensolves, Cholesky QR, small FP64 products, right-operand conversion, mixed digits, the MINRES update."""
import numpy as np
import pytest

from gen import problems as G
from oracle import chase_oracle as O
from tests.helpers import dev, host
from tests.test_gpu_residues import bound, hermitian

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2205_02491_gb300 as P
    return P


# blocks of 128 rows and 64 columns, groups of 8 real or 4 complex runs, up to 64 steps
@pytest.mark.parametrize("n,cplx,runs,steps", [(1, False, 1, 1), (3, True, 2, 3), (63, False, 8, 20), (65, True, 5, 25),
                                               (127, True, 4, 25), (129, False, 3, 25), (1000, True, 8, 30),
                                               (1300, False, 1, 64)])
def test_lanczos(pkg, n, cplx, runs, steps):
    g = np.random.default_rng(n)
    A = hermitian(g, n, cplx) / np.sqrt(n)
    L0 = G.gaussian(g, (n, runs), cplx)
    ne = max(1, n // 10)
    ref = O.lanczos_bounds(A, L0, steps, ne)
    out = pkg.Chase(n, ne, complex_=cplx).lanczos(dev(A), ne, dev(L0), runs, steps)
    for key, val in (("b_sup", ref.b_sup), ("mu_1", ref.mu_1), ("mu_ne", ref.mu_ne), ("theta_max", ref.theta_max)):
        assert abs(out[key] - val) <= 1e-10 * max(1.0, abs(val)), key


# one block to 64, a grid-wide sweep to 127, block Jacobi from 128; blocks of 32
@pytest.mark.parametrize("cplx", [True, False])
@pytest.mark.parametrize("k", [7, 8, 31, 32, 33, 63, 64, 65, 127, 128, 129])
def test_rayleigh_ritz_sizes(pkg, cplx, k):
    n = 300
    g = np.random.default_rng(k)
    A = hermitian(g, n, cplx) / np.sqrt(2 * n)
    Q, _ = np.linalg.qr(G.gaussian(g, (n, k), cplx))
    wo, _ = O.rayleigh_ritz(A, Q)
    Qt = dev(Q)
    w, r = pkg.Chase(n, k, complex_=cplx).rayleigh_ritz(dev(A), Qt)
    V = host(Qt)
    assert np.max(np.abs(w - wo)) <= 1e-12
    assert np.max(np.abs(np.linalg.norm(A @ V - V * w[None, :], axis=0) - r)) <= 1e-11
    assert np.max(np.abs(np.conj(V.T) @ V - np.eye(k))) <= 1e-12


# panels of 16 columns, outer blocks of 128; CUDA-core and tensor-core products
@pytest.mark.parametrize("cplx", [True, False])
@pytest.mark.parametrize("k,l", [(15, 0), (16, 3), (17, 0), (127, 5), (128, 0), (129, 16), (300, 0), (300, 37)])
def test_qr_sizes(pkg, cplx, k, l):
    n = 701
    g = np.random.default_rng(10 * k + l)
    Y = np.linalg.qr(G.gaussian(g, (n, l), cplx))[0] if l else np.zeros((n, 0))
    X = G.gaussian(g, (n, k - l), cplx) * np.exp(g.uniform(-3, 3, size=k - l))[None, :]
    Xt = dev(np.concatenate([Y, X], axis=1))
    pkg.Chase(n, k, complex_=cplx).qr(Xt, nlocked=l)
    Q = host(Xt)
    assert np.array_equal(Q[:, :l], Y)
    assert np.max(np.abs(np.conj(Q.T) @ Q - np.eye(k))) <= 1e-12
    E = X - Q @ (np.conj(Q.T) @ X)
    assert np.all(np.linalg.norm(E, axis=0) <= 1e-11 * np.linalg.norm(X, axis=0))


# tiles of 16 x 16
@pytest.mark.parametrize("cplx", [True, False])
@pytest.mark.parametrize("n,k", [(1, 1), (15, 15), (16, 16), (17, 3), (33, 17), (100, 48)])
def test_small_fp64_products(pkg, cplx, n, k):
    g = np.random.default_rng(100 * n + k)
    A, B = hermitian(g, n, cplx), G.gaussian(g, (n, k), cplx)
    C = host(pkg.Chase(n, k, complex_=cplx).hemm(dev(A), dev(B), "fp64_native"))
    assert np.all(np.abs(C - A @ B) <= 2 * (n + 4) * 2.0 ** -52 * (np.abs(A) @ np.abs(B)))


# clusters of 1, 2, 4 and 8 per column of 512 entries each; one row per combining thread up to 2^19 entries
@pytest.mark.parametrize("n,k,cplx", [(511, 9, False), (513, 9, True), (1024, 9, False), (1025, 9, True), (2049, 9, False),
                                      (4096, 128, False), (4097, 128, False), (4096, 129, True), (4101, 9, True)])
def test_right_operand_columns(pkg, n, k, cplx):
    g = np.random.default_rng(n)
    d, o = g.standard_normal(n), G.gaussian(g, (n,), cplx)
    q = n // 3
    A = np.zeros((n, n), dtype=o.dtype)
    i = np.arange(n - q)
    A[i, i + q], A[i + q, i] = o[i], np.conj(o[i])
    A[np.arange(n), np.arange(n)] = d
    B = G.gaussian(g, (n, k), cplx)
    B[:, 1] = 0.0
    B[:, 2] *= 1e-200
    B[:, 3] *= 1e200
    B[:, 4] *= np.exp(g.uniform(-60, 60, size=n))
    B[n // 2, 5] = np.nan
    C = host(pkg.Chase(n, k, complex_=cplx).hemm(dev(A), dev(B), "fp64"))
    assert np.all(np.isnan(C[:, 5].real)) and np.all(C[:, 1] == 0.0)
    keep = np.arange(k) != 5
    B = B[:, keep]
    ref = d[:, None] * B
    ref[:n - q] += o[:n - q, None] * B[q:]
    ref[q:] += np.conj(o[:n - q, None]) * B[:n - q]
    norms = np.sqrt(d ** 2 + np.pad(np.abs(o[:n - q]) ** 2, (0, q)) + np.pad(np.abs(o[:n - q]) ** 2, (q, 0)))
    scale = np.max(np.abs(B), axis=0)
    scale[scale == 0.0] = 1.0
    nb = np.linalg.norm(B / scale, axis=0) * scale
    tol = 4.0 * np.sqrt(2.0 * n) * 2.0 ** -62 * norms[:, None] * nb[None, :]
    tol += 2.0 ** -50 * (np.abs(d)[:, None] * np.abs(B))
    tol[:n - q] += 2.0 ** -50 * np.abs(o[:n - q, None]) * np.abs(B[q:])
    tol[q:] += 2.0 ** -50 * np.abs(o[:n - q, None]) * np.abs(B[:n - q])
    assert np.all(np.abs(C[:, keep] - ref) <= tol)


# digits of both operands: a product keeps the exact bound of its slices over magnitudes, zeros, subnormals and ties
@pytest.mark.parametrize("mode,rel", [("bf16x3", 2.0 ** -13), ("bf16x6", 2.0 ** -20)])
@pytest.mark.parametrize("n,cplx", [(255, True), (513, False), (1100, True)])
def test_mixed_digits(pkg, mode, rel, n, cplx):
    g = np.random.default_rng(n)
    A = hermitian(g, n, cplx)
    k = 12
    B = G.gaussian(g, (n, k), cplx)
    B[:, 1] = 0.0
    B[:, 2] *= 1e-310
    B[:, 3] *= 1e300
    B[:, 4] = np.round(B[:, 4].real * 256) / 256 + 2.0 ** -10     # ties of the first digit
    B[:, 5] *= np.exp(g.uniform(-30, 0, size=n))
    B[0, 6] = np.inf
    C = host(pkg.Chase(n, k, complex_=cplx).hemm(dev(A), dev(B), mode))
    assert np.all(C[:, 1] == 0.0) and not np.any(np.isfinite(C[:, 6].real))
    for j in (0, 3, 4, 5, 7, 11):
        s = np.max(np.abs(B[:, j]))
        err = np.abs(C[:, j] / s - A @ (B[:, j] / s))
        assert np.all(err <= rel * np.linalg.norm(A, axis=1) * np.linalg.norm(B[:, j] / s)), j


def test_backward_past_the_register_rows(pkg):
    """n > 4096: the MINRES update's entries past the four that a thread keeps in registers."""
    import torch
    n, nev = 4200, 3
    g = np.random.default_rng(5)
    lam = np.concatenate([-1.0 + 0.05 * np.arange(nev + 3), np.sort(g.uniform(-0.6, 1.0, n - nev - 3))])
    p = G.problem_small(n, nev, 9, complex_=False, k_reflect=4, lam=lam, seed_pid=5, cfg=10)
    A = torch.from_numpy(p.dense()).cuda()
    w = torch.tensor([0.3, -1.1, 0.7], dtype=torch.float64, device="cuda")
    C = torch.from_numpy(g.standard_normal((n, nev))).cuda()
    s = pkg.Chase(n, p.ne, complex_=False)
    Ar = A.clone().requires_grad_(True)
    l, V = pkg.ChaseEigh.apply(Ar, s, nev, 9, 1e-12, p.deg, "fp64", dev(p.V0), dev(p.L0), 1e-12, 20000)
    # sign-free loss: w . lambda + sum (V_j . C_j)^2
    ((w * l).sum() + ((V * C).sum(0) ** 2).sum()).backward()
    e, U = torch.linalg.eigh(A)
    gV = 2.0 * (U[:, :nev] * C).sum(0) * C
    M = U.T @ gV
    F = 1.0 / (e[None, :nev] - e[:, None]).masked_fill(torch.eye(n, nev, dtype=torch.bool, device="cuda"), float("inf"))
    ref = U @ (F * M + torch.eye(n, nev, dtype=torch.float64, device="cuda") * w) @ U[:, :nev].T
    ref = 0.5 * (ref + ref.T)
    assert (Ar.grad - ref).abs().max().item() <= 1e-8 * ref.abs().max().item()
