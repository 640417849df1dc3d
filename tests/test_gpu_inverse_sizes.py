"""Inverses and pivots at the edges of the elimination kernels' row and column
splits (one row per warp pass, 32 columns per lane step, CTAs and clusters by
size), on a system that is a single root block; and the solve's iteration as a
graph replay against plain launches."""
import numpy as np
import pytest
import scipy.linalg as sla

import workloads as W

pytestmark = pytest.mark.gpu

U32, U64 = 2.0 ** -24, 2.0 ** -53


@pytest.fixture(scope="module")
def B():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2502_02395_gb300 import build as bld
    bld.build()
    from paper_2502_02395_gb300 import binding
    return binding


@pytest.mark.parametrize("n", [2, 31, 32, 33, 64, 65, 127, 128, 129, 192, 200, 255, 256])
def test_root_inverse(B, n):
    """FP32 elimination: relative error <= 2 n u32 cond (n u backward error of
    elimination); FP64 elimination of the FP32 block: <= 8 u32 and LAPACK's
    pivots; the FP64 factorization: <= 2 n u64 cond and LAPACK's pivots."""
    P = W.cube_points(n, 7)
    S = B.H2Solver.build(P, kernel="laplace_eps", diag_shift=0.1, leaf=256, eta=1.0, tol=1e-8, far_samples=64,
                         near_samples=8)
    assert S.stats()["levels"][0]["D"] == n
    for prec, rr in (("fp16", 0), ("fp16", 1), ("fp64", 0)):
        S.set_option("rr_lu_fp64", rr)
        S.factor(prec)
        A = S.export("A", 0).reshape(n, n).astype(np.float64)
        inv = S.export("root_inv", 0).reshape(n, n).astype(np.float64)
        ref = np.linalg.inv(A)
        e = np.linalg.norm(inv - ref) / np.linalg.norm(ref)
        u = U64 if prec == "fp64" else U32
        assert e <= (8 * U32 if rr else 2 * max(n, 8) * u * np.linalg.cond(A)), (prec, rr, e)
        if rr or prec == "fp64":
            assert (S.export("root_piv", 0) == sla.lu_factor(A)[1]).all(), (prec, rr)


@pytest.mark.parametrize("n,leaf,prec", [(700, 49, "bf16"), (2048, 256, "fp16"), (5000, 64, "fp16")])
def test_graph_replay_and_launches(B, n, leaf, prec):
    """The same solve with and without graph replay: both reach the target, in
    as many iterations, and differ by no more than two such residuals."""
    P = W.cube_points(n, 9)
    S = B.H2Solver.build(P, kernel="yukawa_eps", diag_shift=1.0, leaf=leaf, eta=1.0, tol=1e-8, far_samples=512,
                         near_samples=32)
    b = W.uniform_rhs(n, 10)
    out = []
    for g in (0, 1):
        S.set_option("graphs", g)
        S.factor(prec)
        x, rel, its = S.solve(b, target=1e-10, max_iters=100)
        assert rel <= 1e-10
        out.append((x, its))
    assert out[0][1] == out[1][1]
    assert np.linalg.norm(S.matvec(out[0][0] - out[1][0])) <= 2e-10 * np.linalg.norm(b)
