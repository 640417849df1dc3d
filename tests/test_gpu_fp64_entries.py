"""FP64 factorizations entry by entry: blocks whose entries range over many
decades (a Gaussian kernel of short length: from 1 to 1e-80 within a row) and
diagonals far above the other entries.  Every entry of a projected block is as
accurate as FP64 sums of its own terms are, not only the block in its norm."""
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


@pytest.mark.parametrize("n,leaf,rank,kw", [
    (512, 64, 32, dict(kernel="gaussian", ell=0.05, diag_shift=1.0)),
    (512, 64, 32, dict(kernel="yukawa_eps", diag_shift=1e8)),
    (600, 75, 31, dict(kernel="gaussian", ell=0.05, diag_shift=1.0)),
    (130, 33, 8, dict(kernel="gaussian", ell=0.1, diag_shift=1.0)),
    (130, 33, 8, dict(kernel="yukawa_eps", diag_shift=1e8))])
def test_projected_blocks_entry_by_entry(B, n, leaf, rank, kw):
    """Ahat_ij = U_i A_ij U_j^T in FP64 against the same products in extended
    precision: a running sum of D products is within D u of the sum of their
    sizes (two products: |dW| <= D u |A||U^T|, then |U||dW| + D u |U||W|; 1 % for
    terms of u^2; entries below 1e-290 are left to underflow)."""
    from oracle.construct import construct
    from oracle.instance import flatten
    from oracle.kernels import Kernel
    name = kw["kernel"]
    kk = {k: v for k, v in kw.items() if k != "kernel"}
    flat = flatten(construct(W.cube_points(n, 3), Kernel(name, **kk), leaf, 1.0, 1e-12, rank, 0, 0))
    S = B.H2Solver.from_instance(flat, leaf=leaf, eta=1.0, tol=1e-12, max_rank=rank, far_samples=0, near_samples=0, **kw)
    L, D, K = flat["L"], int(flat["D"][-1]), int(flat["K"][-1])
    R = D - K
    S.factor("fp64")
    U = S.export("U", L).reshape(-1, D, D)
    A = S.export("A", L).reshape(-1, D, D)
    got = S.export("Ahat", L).reshape(-1, D, D)
    for q, (i, j) in list(enumerate(flat["near"][L]))[:10]:
        Wx = A[q].astype(np.longdouble) @ U[j].T.astype(np.longdouble)
        ref = (U[i].astype(np.longdouble) @ Wx).astype(np.float64)
        size = np.abs(U[i]) @ (np.abs(A[q]) @ np.abs(U[j]).T) + np.abs(U[i]) @ np.abs(Wx.astype(np.float64))
        err = np.abs(got[q] - ref)
        if i == j:
            err[R:, R:] = 0.0  # (holds the Schur update)
        assert (err <= 1.01 * D * U64 * size + 1e-290).all(), (i, j)
