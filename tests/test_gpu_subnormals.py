"""Products with operands whose entries are all subnormal: scaled without loss by exact powers of two, FP64-class and
mixed."""
import numpy as np
import pytest

from gen import problems as G
from tests.helpers import dev, host
from tests.test_gpu_residues import bound, exact, hermitian

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2205_02491_gb300 as P
    return P


def small_columns(g, n, k, cplx):
    """Columns of subnormal numbers (the first pair's largest are just above), and the same times 2^1000, exactly."""
    scale = np.array([2.0 ** e for e in (-1029, -1030, -1035, -1045, -1060)])[np.arange(k) % 5]
    B = G.gaussian(g, (n, k), cplx) * scale[None, :]
    return B, B * 2.0 ** 1000


# columns by right_planes_kernel
@pytest.mark.parametrize("cplx", [True, False])
@pytest.mark.parametrize("n,k", [(65, 7), (700, 10)])
def test_fp64_product_of_subnormal_columns(pkg, n, k, cplx):
    g = np.random.default_rng(n)
    A = hermitian(g, n, cplx)
    B, Bs = small_columns(g, n, k, cplx)
    C = host(pkg.Chase(n, k, complex_=cplx).hemm(dev(A * 2.0 ** 990), dev(B), "fp64"))
    ref = exact(A, Bs)
    assert np.all(np.abs(C * 2.0 ** 10 - ref) <= bound(A, Bs, ref))


# rows of a subnormal A (col_exponent_kernel) against large columns
@pytest.mark.parametrize("cplx", [True, False])
def test_fp64_product_of_a_subnormal_matrix(pkg, cplx):
    n, k = 300, 9
    g = np.random.default_rng(3)
    A = hermitian(g, n, cplx) * 2.0 ** -1032
    A = np.tril(A) + np.conj(np.tril(A, -1)).T
    B = G.gaussian(g, (n, k), cplx)
    C = host(pkg.Chase(n, k, complex_=cplx).hemm(dev(A), dev(B * 2.0 ** 990), "fp64"))
    ref = exact(A * 2.0 ** 1000, B)
    assert np.all(np.abs(C * 2.0 ** 10 - ref) <= bound(A * 2.0 ** 1000, B, ref))


@pytest.mark.parametrize("mode,rel", [("bf16x3", 2.0 ** -13), ("bf16x6", 2.0 ** -20)])
@pytest.mark.parametrize("n,cplx", [(255, True), (513, False)])
def test_mixed_product_of_subnormal_columns(pkg, mode, rel, n, cplx):
    g = np.random.default_rng(n)
    A = hermitian(g, n, cplx)
    k = 10
    B, Bs = small_columns(g, n, k, cplx)
    C = host(pkg.Chase(n, k, complex_=cplx).hemm(dev(A * 2.0 ** 990), dev(B), mode)) * 2.0 ** 10
    s = np.max(np.abs(Bs), axis=0)
    err = np.abs(C / s - A @ (Bs / s))
    assert np.all(err <= rel * np.linalg.norm(A, axis=1)[:, None] * np.linalg.norm(Bs / s, axis=0)[None, :])
