"""Rayleigh-Ritz of quotients with eigenvalues closer than the FP32 first pass tells apart: groups spaced around the
line (1e-5 of the norm) below which a pair is solved as part of a cluster."""
import numpy as np
import pytest

from tests.helpers import dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2205_02491_gb300 as P
    return P


def spectrum(g, k, m, spacing):
    """k values on [-1, 1], about evenly spread, m of them `spacing` apart, the norm 1."""
    lam = np.linspace(-1.0, 1.0, k) + g.uniform(-0.3, 0.3, k) * 2.0 / k
    lam /= np.max(np.abs(lam))
    at = g.integers(0, k - m)
    lam[at:at + m] = lam[at] + spacing * np.arange(m)
    return np.sort(lam)


# one block, a grid-wide sweep and block Jacobi
@pytest.mark.parametrize("cplx", [True, False])
@pytest.mark.parametrize("k", [8, 24, 48, 63, 100, 200])
def test_rayleigh_ritz_of_close_eigenvalues(pkg, cplx, k):
    import torch
    n = 3 * k + 5
    g = np.random.default_rng(k)
    dt = torch.complex128 if cplx else torch.float64
    gen = torch.Generator(device="cuda").manual_seed(k)
    rand = lambda a, b: torch.randn((a, b), generator=gen, device="cuda", dtype=dt)  # noqa: E731
    U = torch.linalg.qr(rand(n, n))[0]
    s = pkg.Chase(n, k, complex_=cplx)
    worst = np.zeros(3)
    for m in (2, 3, 4):
        for spacing in (5e-7, 9e-6, 1.05e-5, 1.5e-5, 2e-5, 3e-5):
            for _ in range(6):
                lam = spectrum(g, k, m, spacing)
                rest = dev(np.concatenate([lam, g.uniform(-1.0, 1.0, n - k)]))
                A = (U * rest[None, :]) @ U.mH
                A = 0.5 * (A + A.mH)
                Q = U[:, :k] @ torch.linalg.qr(rand(k, k))[0]
                Qt = Q.mT.contiguous()
                w, r = s.rayleigh_ritz(A.mT.contiguous(), Qt)
                V = Qt.mT
                wt = torch.from_numpy(w).cuda()
                worst = np.maximum(worst, [np.max(np.abs(w - lam)),
                                           torch.linalg.vector_norm(A @ V - V * wt[None, :], dim=0).max().item(),
                                           (V.mH @ V - torch.eye(k, dtype=dt, device="cuda")).abs().max().item()])
    # eigenvalues, residuals (the block spans an invariant subspace) and orthonormality of a quotient of norm 1
    assert np.all(worst <= 1e-12), worst
