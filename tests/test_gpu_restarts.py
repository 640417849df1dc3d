"""Restart lengths that change between solves of one context: the host's reads of
an inner iteration's numbers do not depend on what an earlier solve left in
their place."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2502_02395_gb300 import build as bld
    bld.build()
    from paper_2502_02395_gb300 import binding
    return binding


def context(B, n):
    return B.H2Solver.build(W.cube_points(n, 3), kernel="yukawa_eps", eps=0.05, leaf=128, eta=1.0, tol=1e-12, max_rank=64,
                            far_samples=256, near_samples=32)


@pytest.mark.parametrize("graphs", [1, 0])
def test_restarts_on_one_context(B, graphs):
    """Solves at restarts 30, 10, 20, 25 and 30 on one context: iteration counts
    and residual histories of fresh contexts (the same launches on the same
    numbers; the history's residuals to 1e-6 of themselves)."""
    n = 4096
    b = W.uniform_rhs(n, 6)
    S = context(B, n)
    S.set_option("graphs", graphs)
    S.factor("bf16")
    for restart in (30, 10, 20, 25, 30):
        S.set_refinement("auto", restart)
        x, rel, its = S.solve(b, target=1e-10, max_iters=300)
        hist = S.stats()["history"]
        F = context(B, n)
        F.set_option("graphs", graphs)
        F.factor("bf16")
        F.set_refinement("auto", restart)
        xf, relf, itsf = F.solve(b, target=1e-10, max_iters=300)
        assert itsf > 13 and its == itsf, restart
        assert np.allclose(hist, F.stats()["history"], rtol=1e-6, atol=0), restart
        assert np.linalg.norm(x - xf) <= 1e-9 * np.linalg.norm(xf)
        F.close()


def test_launch_count_with_threads(B):
    """Contexts whose solves are captured and replayed in four threads at a time
    count as many launches as one after another."""
    import threading
    sizes = [1024, 1500, 2048, 3000]
    ctx = lambda n: context(B, n)

    def work(S, n):
        S.factor("fp16")
        for k in range(3):
            S.solve(W.uniform_rhs(n, k), target=1e-10, max_iters=300)

    def count(threads):
        solvers = [(ctx(n), n) for n in sizes]
        n0 = solvers[0][0].stats()["kernel_launches"]
        ts = [threading.Thread(target=work, args=s) for s in solvers]
        for t in ts:
            t.start()
            if not threads:
                t.join()
        for t in ts:
            t.join()
        n1 = solvers[0][0].stats()["kernel_launches"]
        for S, _ in solvers:
            S.close()
        return n1 - n0

    one = count(False)
    for _ in range(5):
        assert count(True) == one
