"""FP64-class products through residues on the GPU: tile edges, worst-case chunk sums, non-finite operands, and A's
planes converted in passes when memory is short."""
import numpy as np
import pytest

from gen import problems as G
from tests.helpers import dev, host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2205_02491_gb300 as P
    return P


def hermitian(g, n, cplx):
    X = G.gaussian(g, (n, n), cplx)
    return 0.5 * (X + np.conj(X.T))


def exact(A, B):
    ld = np.longdouble
    if not np.iscomplexobj(A):
        return (A.astype(ld) @ B.astype(ld)).astype(np.float64)
    Ar, Ai, Br, Bi = A.real.astype(ld), A.imag.astype(ld), B.real.astype(ld), B.imag.astype(ld)
    return (Ar @ Br - Ai @ Bi).astype(np.float64) + 1j * (Ar @ Bi + Ai @ Br).astype(np.float64)


def bound(A, B, ref):
    """Operands are rounded to half a unit of 2^-62 of a power of two at most twice their vector's norm; the result and
    its reference are rounded to FP64."""
    K = A.shape[1]
    na, nb = np.linalg.norm(A, axis=1), np.linalg.norm(B, axis=0)
    return 4.0 * np.sqrt(2.0 * K) * 2.0 ** -62 * na[:, None] * nb[None, :] + 2.0 ** -51 * np.abs(ref)


# tiles of 256 rows (128 per CTA of a pair), columns in blocks of 32 up to 256, K in blocks of 64 and chunks of 1024
@pytest.mark.parametrize("cplx", [True, False])
@pytest.mark.parametrize("n,k", [(1, 1), (63, 31), (64, 32), (65, 33), (127, 1), (128, 127), (129, 128), (255, 129),
                                 (256, 255), (257, 256), (513, 257), (700, 300), (1023, 40), (1025, 5)])
def test_tile_edges(pkg, cplx, n, k):
    g = np.random.default_rng(1000 * n + k)
    A = hermitian(g, n, cplx)
    B = G.gaussian(g, (n, k), cplx) * np.exp(g.uniform(-40, 40, size=k))[None, :]
    s = pkg.Chase(n, max(1, min(k, n)), complex_=cplx)
    for j in range(0, k, n):
        Bj = B[:, j:j + n]
        C = host(s.hemm(dev(A), dev(Bj), "fp64"))
        ref = exact(A, Bj)
        assert np.all(np.abs(C - ref) <= bound(A, Bj, ref))


def test_chunk_sums_at_their_largest(pkg):
    """Entries 1 + 2^-49 scale to 2^56 + 2^7: residues of +-128 modulo 256 everywhere, so the chunk sum modulo that
    modulus is 2^24, the largest exact FP32 value it can take."""
    n, k = 1024, 40
    x = 1.0 + 2.0 ** -49
    A = np.full((n, n), x)
    s = pkg.Chase(n, k, complex_=False)
    C = host(s.hemm(dev(A), dev(np.full((n, k), x)), "fp64"))
    # n x^2 = 1024 + 2^-38 + 2^-88, rounded to 2^-42
    assert np.array_equal(C, np.full((n, k), 1024.0 + 2.0 ** -38))


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_operands_mark_their_rows_and_columns(pkg, bad):
    n, k = 200, 20
    g = np.random.default_rng(4)
    A, B = hermitian(g, n, True), G.gaussian(g, (n, k), True)
    A[7, 30] = bad
    A[30, 7] = bad
    B[11, 5] = bad
    s = pkg.Chase(n, k, complex_=True)
    C = host(s.hemm(dev(A), dev(B), "fp64"))
    off = np.zeros((n, k), bool)
    off[[7, 30], :] = True
    off[:, 5] = True
    assert np.all(np.isnan(C[off]))
    fin = ~off
    ref = np.nan_to_num(A, nan=0.0, posinf=0.0) @ np.nan_to_num(B, nan=0.0, posinf=0.0)
    assert np.all(np.abs(C[fin] - ref[fin]) <= 1e-12 * np.abs(ref[fin]).max())


def test_extreme_magnitudes(pkg):
    """Norms whose squares overflow or underflow take the scaled pass; zero columns give zeros."""
    n, k = 150, 6
    g = np.random.default_rng(6)
    A, B = hermitian(g, n, False), G.gaussian(g, (n, k), False)
    B[:, 1] = 0.0
    B[:, 2] *= 1e-200
    B[:, 3] *= 1e200
    s = pkg.Chase(n, k, complex_=False)
    C = host(s.hemm(dev(A), dev(B), "fp64"))
    scale = np.array([1.0, 1.0, 1e200, 1e-200, 1.0, 1.0])
    ref = exact(A, B * scale)
    assert np.all(C[:, 1] == 0.0)
    assert np.all(np.abs(C * scale - ref) <= bound(A, B * scale, ref) + 2.0 ** -50 * np.abs(ref))


def test_same_result_when_memory_holds_part_of_the_planes(pkg):
    """With little device memory free a context keeps fewer residue planes of A and converts them in passes per
    product: same arithmetic, same bits."""
    import torch
    n, k = 6000, 50
    g = torch.Generator(device="cuda:0").manual_seed(3)
    X = torch.randn((n, n), generator=g, dtype=torch.float64, device="cuda:0")
    A = 0.5 * (X + X.mT)
    B = torch.randn((k, n), generator=g, dtype=torch.float64, device="cuda:0")
    s = pkg.Chase(n, k, complex_=False)
    C = s.hemm(A, B, "fp64")
    s.close()
    del X
    torch.cuda.empty_cache()
    need = pkg.workspace_bytes(n, k, complex_=False)
    free, _ = torch.cuda.mem_get_info()
    hold = torch.empty(free - need - (400 << 20), dtype=torch.uint8, device="cuda:0")
    try:
        s = pkg.Chase(n, k, complex_=False)
        D = s.hemm(A, B, "fp64")
        s.close()
    finally:
        del hold
        torch.cuda.empty_cache()
    assert torch.equal(C, D)
