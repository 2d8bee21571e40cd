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


@pytest.mark.parametrize("cplx", [True, False])
@pytest.mark.parametrize("n,runs", [(63, 1), (129, 3), (700, 4), (1300, 8)])
def test_native_mode_rests_on_no_tensor_core_product(pkg, cplx, n, runs):
    """The native mode is the reference for the others: with every wait of the product kernel run out it still solves."""
    p = G.problem_small(n, 8, 6, complex_=cplx, seed_pid=11)
    s = pkg.Chase(n, p.ne, complex_=cplx, opts={"lanczos_runs": runs})
    L0 = G.gaussian(np.random.default_rng(n), (n, runs), cplx)
    A, V0, L0 = dev(p.dense()), dev(p.V0), dev(L0)
    ref = s.lanczos(A, p.ne, L0, runs, 25)
    pkg.set_wait_limit_ns(1)
    try:
        w, _ = s.solve(A, p.nev, p.nex, p.tol, p.deg, "fp64_native", V0, L0)
    finally:
        pkg.set_wait_limit_ns(0)
    st = s.stats()
    assert np.max(np.abs(w.cpu().numpy() - p.lam[:p.nev])) <= 1e-10 * p.norm2()
    for key in ("b_sup", "mu_1"):
        assert abs(st[key] - ref[key]) <= 1e-10 * p.norm2(), key


@pytest.mark.parametrize("n_max,n,runs,steps", [(16000, 8000, 8, 40), (20000, 20000, 2, 64), (20000, 300, 8, 64)])
def test_settings_other_than_the_contexts(pkg, n_max, n, runs, steps):
    """A context made for 4 runs of 25 steps also takes more steps of fewer runs, or more of both at a smaller n."""
    import torch
    gen = torch.Generator(device="cuda").manual_seed(n)
    X = torch.randn((n, n), generator=gen, device="cuda", dtype=torch.float64)
    A = X.add_(X.mT.clone()).mul_(0.5)
    L0 = torch.randn((runs, n), generator=gen, device="cuda", dtype=torch.float64)
    s = pkg.Chase(n_max, 8, complex_=False)
    out = s.lanczos(A, 8, L0, runs, steps)
    s.close()
    s = pkg.Chase(n, 8, complex_=False, opts={"lanczos_runs": runs, "lanczos_steps": steps})
    assert s.lanczos(A, 8, L0, runs, steps) == out
    s.close()
