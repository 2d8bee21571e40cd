"""Device memory that is short: what contexts hold beyond their needs gives way to other contexts, batches and calls."""
import threading

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


def test_contexts_created_together(pkg):
    """Both needs and the half of the rest that one of them takes fit; what both would take of it does not."""
    import torch
    n, k = 16000, 64
    need = pkg.workspace_bytes(n, k, complex_=False)
    g = torch.Generator(device="cuda").manual_seed(1)
    X = torch.randn((n, n), generator=g, device="cuda", dtype=torch.float64)
    A = X.add_(X.mT.clone()).mul_(0.5)
    B = torch.randn((k, n), generator=g, device="cuda", dtype=torch.float64)
    s = pkg.Chase(n, k, complex_=False)
    C = s.hemm(A, B, "fp64")
    s.close()
    torch.cuda.empty_cache()
    torch.cuda.synchronize()
    free, _ = torch.cuda.mem_get_info()
    hold = torch.empty(free - 3 * need - (1 << 30), dtype=torch.uint8, device="cuda")
    try:
        for _ in range(10):
            made, failed = [], []
            start = threading.Barrier(2)

            def create():
                start.wait()
                try:
                    made.append(pkg.Chase(n, k, complex_=False))
                except pkg.ChaseError as e:
                    failed.append(e)

            threads = [threading.Thread(target=create) for _ in range(2)]
            for t in threads:
                t.start()
            for t in threads:
                t.join()
            assert not failed, failed
            for s in made:
                assert torch.equal(s.hemm(A, B, "fp64"), C)
                s.close()
    finally:
        del hold
        torch.cuda.empty_cache()


def test_batch_takes_back_what_its_context_holds(pkg):
    """The batch context holds all of A's planes for its largest size; a batch whose workspaces do not fit beside them
    takes them back."""
    import torch
    from gen import problems as G
    from tests.helpers import dev
    probs = [G.problem_small(n, 10, 6, complex_=False, seed_pid=30 + i) for i, n in enumerate((1800, 2100))]
    n_max, ne = 14000, max(p.ne for p in probs)
    need = sum(pkg.workspace_bytes(p.n, p.ne, complex_=False) for p in probs)
    args = lambda: ([dev(p.dense()) for p in probs], [p.nev for p in probs], [p.nex for p in probs], 1e-10, 20, "fp64",  # noqa: E731
                    [dev(p.V0) for p in probs], [dev(p.L0) for p in probs])
    a = args()
    s = pkg.Chase(n_max, ne, complex_=False)
    torch.cuda.empty_cache()
    torch.cuda.synchronize()
    free, _ = torch.cuda.mem_get_info()
    hold = torch.empty(free - need // 2 - (64 << 20), dtype=torch.uint8, device="cuda")
    try:
        w, _ = s.solve_batched(*a)
    finally:
        del hold
        torch.cuda.empty_cache()
    for p, wp in zip(probs, w):
        assert abs(wp.cpu().numpy() - p.lam[:p.nev]).max() <= 1e-10 * p.norm2()
    # the context's own planes are the fewest now: same result as any other context's
    v0, l0 = torch.randn((ne, 2100), dtype=torch.float64, device="cuda"), a[7][1]
    w1, _ = s.solve(a[0][1], probs[1].nev, probs[1].nex, 1e-10, 20, "fp64", v0, l0)
    assert abs(w1.cpu().numpy() - probs[1].lam[:probs[1].nev]).max() <= 1e-10 * probs[1].norm2()
    s.close()


def test_new_contexts_come_before_planes_of_others(pkg):
    """Three contexts whose needs fit: what the first two hold beyond theirs gives way to the third, also while another
    thread's calls use one of them; products keep their bits."""
    import torch
    n, k = 12000, 48
    need = pkg.workspace_bytes(n, k, complex_=False)
    g = torch.Generator(device="cuda").manual_seed(2)
    X = torch.randn((n, n), generator=g, device="cuda", dtype=torch.float64)
    A = X.add_(X.mT.clone()).mul_(0.5)
    B = torch.randn((k, n), generator=g, device="cuda", dtype=torch.float64)
    first = pkg.Chase(n, k, complex_=False)
    C = first.hemm(A, B, "fp64")
    first.close()
    torch.cuda.empty_cache()
    torch.cuda.synchronize()
    free, _ = torch.cuda.mem_get_info()
    hold = torch.empty(free - 3 * need - (512 << 20), dtype=torch.uint8, device="cuda")
    made = []
    try:
        for _ in range(3):
            made.append(pkg.Chase(n, k, complex_=False))
        for s in made:
            assert torch.equal(s.hemm(A, B, "fp64"), C)
        made.pop().close()
        stop, wrong = threading.Event(), []

        def use():
            while not stop.is_set():
                if not torch.equal(made[0].hemm(A, B, "fp64"), C):
                    wrong.append(1)

        t = threading.Thread(target=use)
        t.start()
        for _ in range(10):
            try:
                pkg.Chase(n, k, complex_=False).close()
            except pkg.ChaseError as e:  # the context in use kept its planes
                assert e.status == 2
        stop.set()
        t.join()
        assert not wrong
    finally:
        for s in made:
            s.close()
        del hold
        torch.cuda.empty_cache()


def test_copy_of_a_host_matrix_comes_before_planes(pkg):
    """The device copy of a host A takes the place of planes where there is no other room."""
    import torch
    from gen import problems as G
    p = G.problem_small(5000, 8, 6, complex_=False, seed_pid=40)
    A, V0, L0 = (torch.from_numpy(np.ascontiguousarray(x.T)) for x in (p.dense(), p.V0, p.L0))
    s = pkg.Chase(9000, p.ne, complex_=False)
    torch.cuda.empty_cache()
    torch.cuda.synchronize()
    free, _ = torch.cuda.mem_get_info()
    hold = torch.empty(free - (150 << 20), dtype=torch.uint8, device="cuda")
    try:
        w, _ = s.solve(A, p.nev, p.nex, 1e-10, 20, "fp64", V0, L0)
    finally:
        del hold
        torch.cuda.empty_cache()
    assert np.max(np.abs(w.numpy() - p.lam[:p.nev])) <= 1e-10 * p.norm2()
    s.close()
