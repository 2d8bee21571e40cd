"""Lanczos bounds at the ends of what they take: non-finite inputs, waits that run out, the native mode, and settings
other than the context's."""
import numpy as np
import pytest

from gen import problems as G
from tests.helpers import dev
from tests.test_gpu_residues import hermitian

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2205_02491_gb300 as P
    return P


# one entry of A (every run meets it), one start vector of four
@pytest.mark.parametrize("cplx", [True, False])
@pytest.mark.parametrize("where", ["A", "L0", "zero start"])
def test_non_finite_sums_are_an_error(pkg, cplx, where):
    n, runs = 200, 4
    g = np.random.default_rng(1)
    A, L0 = hermitian(g, n, cplx), G.gaussian(g, (n, runs), cplx)
    s = pkg.Chase(n, 20, complex_=cplx)
    good = s.lanczos(dev(A), 20, dev(L0), runs, 25)  # leaves finite Ritz values in the context
    if where == "A":
        A[7, 30] = A[30, 7] = np.nan
    elif where == "L0":
        L0[11, 2] = np.nan
    else:
        L0[:, 2] = 0.0
    with pytest.raises(pkg.ChaseError) as e:
        s.lanczos(dev(A), 20, dev(L0), runs, 25)
    assert e.value.status == 5
    A, L0 = np.nan_to_num(A), np.nan_to_num(L0)
    L0[:, 2] += 1.0
    assert all(np.isfinite(v) for v in s.lanczos(dev(A), 20, dev(L0), runs, 25).values()) and good["b_sup"] > 0.0


@pytest.mark.parametrize("cplx", [True, False])
def test_waits_that_run_out_are_a_timeout(pkg, cplx):
    """With the wait limit at 1 ns a wait of the product kernel gives up: the call reports it and the context stays
    usable."""
    n, runs = 1500, 4
    g = np.random.default_rng(2)
    A, L0 = dev(hermitian(g, n, cplx)), dev(G.gaussian(g, (n, runs), cplx))
    s = pkg.Chase(n, 20, complex_=cplx)
    ref = s.lanczos(A, 20, L0, runs, 25)
    pkg.set_wait_limit_ns(1)
    try:
        with pytest.raises(pkg.ChaseError) as e:
            s.lanczos(A, 20, L0, runs, 25)
        assert e.value.status == 8
        with pytest.raises(pkg.ChaseError) as e:
            s.solve(A, 12, 8, 1e-10, 20, "fp64", None, L0)
        assert e.value.status == 8
    finally:
        pkg.set_wait_limit_ns(0)
    assert s.lanczos(A, 20, L0, runs, 25) == ref


def test_sweep_wait_limit(pkg):
    """The grid barrier of the Jacobi sweep (65 to 127 columns) reports a wait that runs out too."""
    n, k = 400, 96
    g = np.random.default_rng(3)
    A = dev(hermitian(g, n, True))
    Q = dev(np.linalg.qr(G.gaussian(g, (n, k), True))[0])
    s = pkg.Chase(n, k, complex_=True)
    pkg.set_wait_limit_ns(1)
    try:
        with pytest.raises(pkg.ChaseError) as e:
            s.rayleigh_ritz(A, Q.clone())
        assert e.value.status == 8
    finally:
        pkg.set_wait_limit_ns(0)
    w, _ = s.rayleigh_ritz(A, Q.clone())
    assert np.all(np.isfinite(w))
