"""Contexts created at the same time: each counts the same free memory, so what they take beyond their needs must give
way."""
import threading

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
