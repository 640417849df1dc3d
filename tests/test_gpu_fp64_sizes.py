"""FP64 factorizations at the edges of the FP64 kernels' tiles: box dimensions
and ranks below, at and above multiples of 64 and 128, odd ones (no 16-byte
accesses), ranks from tolerances."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

U64 = 2.0 ** -53


@pytest.fixture(scope="module")
def B():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2502_02395_gb300 import build as bld
    bld.build()
    from paper_2502_02395_gb300 import binding
    return binding


# (points, leaf, tolerance, eta)
SIZES = [(60, 33, 1e-6, 1.0), (519, 66, 1e-6, 1.0), (1003, 64, 1e-10, 1.0), (1600, 49, 1e-10, 0.0),
         (2999, 200, 1e-4, 1.0), (4011, 255, 1e-10, 1.0), (4096, 256, 1e-10, 1.0)]


@pytest.mark.parametrize("n,leaf,tol,eta", SIZES)
def test_fp64_bases_and_projection(B, n, leaf, tol, eta):
    """The bases' orthogonality (K reflectors of a few roundings each, 20 K u
    at most) and R of X = U^S R, and the projected diagonal blocks against
    U_i A_ii U_i^T: every entry of a product of inner length D is off by at
    most D 2^-53 (largest entry of the row x of the column), in both products
    and in the reference's, beside the roundings of the results."""
    P = W.cube_points(n, 3)
    S = B.H2Solver.build(P, kernel="yukawa_eps", diag_shift=1.0, leaf=leaf, eta=eta, tol=tol, far_samples=512,
                         near_samples=32)
    st = S.stats()
    L = st["L"]
    S.factor("fp64")
    lv = st["levels"][L]
    nb, D, K = lv["nb"], lv["D"], lv["K"]
    R = D - K
    U = S.export("U", L).reshape(nb, D, D)
    for i in range(nb):
        assert np.abs(U[i] @ U[i].T - np.eye(D)).max() <= 20 * max(K, 1) * U64
    A = S.export("A", L).reshape(-1, D, D)[0]
    got = S.export("Ahat", L).reshape(-1, D, D)[0].copy()
    Wm = A @ U[0].T
    ref = U[0] @ Wm
    got[R:, R:] = ref[R:, R:]  # (holds the Schur update)
    row, col = lambda M: np.abs(M).max(axis=1), lambda M: np.abs(M).max(axis=0)
    dW = D * U64 * np.outer(row(A), col(U[0].T)) + U64 * np.abs(Wm)
    bound = np.abs(U[0]) @ dW + D * U64 * np.outer(row(U[0]), col(Wm)) + U64 * np.abs(ref)
    assert (np.abs(got - ref) <= 2 * bound).all()
    b = W.uniform_rhs(n, 5)
    x = S.solve(b)
    x = x[0] if isinstance(x, tuple) else x
    assert np.linalg.norm(S.matvec(x) - b) <= 1e-9 * np.linalg.norm(b)
