"""Phases of numbers whose squares underflow.  The FP64 Jacobi eigensolver on degenerate spectra: entries between equal
eigenvalues fall far below the square root of the smallest FP64 number while the sweeps go on for the others.  Householder
reflectors: a column whose first entry is that small."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2205_02491_gb300 as P
    return P


SPECTRA = {
    "quartic": lambda k: -1.0 + 2.0 * np.linspace(0.0, 1.0, k) ** 4,
    "half equal": lambda k: np.sort(np.concatenate([np.full(k // 2, -1.0), np.linspace(-0.9, 1.0, k - k // 2)])),
    "two values": lambda k: np.sort(np.where(np.arange(k) % 3 == 0, -1.0, 0.5)),
}


@pytest.mark.parametrize("cplx", [True, False])
@pytest.mark.parametrize("k", [40, 200, 437, 500])
@pytest.mark.parametrize("spectrum", sorted(SPECTRA))
def test_jacobi_keeps_its_vectors_orthonormal(pkg, cplx, k, spectrum):
    import torch
    dt = torch.complex128 if cplx else torch.float64
    gen = torch.Generator(device="cuda").manual_seed(k)
    lam = torch.from_numpy(SPECTRA[spectrum](k)).cuda()
    s = pkg.Chase(k, k, complex_=cplx)
    for _ in range(3):
        P = torch.linalg.qr(torch.randn((k, k), generator=gen, device="cuda", dtype=dt))[0]
        G = (P * lam[None, :]) @ P.mH
        G = 0.5 * (G + G.mH)
        w, Zt = s.heevj(G.mT.contiguous())
        Z, wt = Zt.mT, torch.from_numpy(w).cuda()
        assert (wt - lam).abs().max().item() <= 1e-12
        assert torch.linalg.vector_norm(G @ Z - Z * wt[None, :], dim=0).max().item() <= 1e-12
        assert (Z.mH @ Z - torch.eye(k, dtype=dt, device="cuda")).abs().max().item() <= 1e-12


@pytest.mark.parametrize("cplx,k", [(True, 200), (False, 437)])
def test_rayleigh_ritz_of_a_degenerate_quotient(pkg, cplx, k):
    """Groups of more columns than a cluster takes go to the FP64 solver; smaller ones are solved as clusters."""
    import torch
    n = 3 * k + 5
    dt = torch.complex128 if cplx else torch.float64
    gen = torch.Generator(device="cuda").manual_seed(k)
    rand = lambda a, b: torch.randn((a, b), generator=gen, device="cuda", dtype=dt)  # noqa: E731
    U = torch.linalg.qr(rand(n, n))[0]
    s = pkg.Chase(n, k, complex_=cplx)
    for group in (2, 16, 32, 33, k // 2):
        lam = np.linspace(-1.0, 1.0, k)
        lam[:group] = -1.0
        rest = torch.from_numpy(np.concatenate([lam, np.linspace(-0.8, 0.9, n - k)])).cuda()
        A = (U * rest[None, :]) @ U.mH
        A = 0.5 * (A + A.mH)
        Qt = (U[:, :k] @ torch.linalg.qr(rand(k, k))[0]).mT.contiguous()
        w, _ = s.rayleigh_ritz(A.mT.contiguous(), Qt)
        V, wt = Qt.mT, torch.from_numpy(w).cuda()
        assert np.max(np.abs(w - lam)) <= 1e-12, group
        assert torch.linalg.vector_norm(A @ V - V * wt[None, :], dim=0).max().item() <= 1e-12, group
        assert (V.mH @ V - torch.eye(k, dtype=dt, device="cuda")).abs().max().item() <= 1e-12, group


@pytest.mark.parametrize("cplx", [True, False])
@pytest.mark.parametrize("exponent", [-160.0, -160.5, -161.0, -161.5, -305.0])
def test_householder_qr_with_a_tiny_first_entry(pkg, cplx, exponent):
    from tests.helpers import dev, host
    n, k = 400, 24
    g = np.random.default_rng(7)
    rand = lambda *shape: g.standard_normal(shape) + (1j * g.standard_normal(shape) if cplx else 0.0)  # noqa: E731
    X = rand(n, k)
    X[:, 9] = X[:, 4] + 1e-13 * rand(n)  # numerically dependent: the block goes to the Householder QR
    X[0] *= 10.0 ** exponent
    s = pkg.Chase(n, k, complex_=cplx)
    before = s.stats()["qr_householder"]
    Xt = dev(X)
    s.qr(Xt)
    assert s.stats()["qr_householder"] == before + 1
    Q = host(Xt)
    assert np.max(np.abs(np.conj(Q.T) @ Q - np.eye(k))) <= 1e-12
    R = X - Q @ (np.conj(Q.T) @ X)
    assert np.max(np.linalg.norm(R, axis=0) / np.linalg.norm(X, axis=0)) <= 1e-10
