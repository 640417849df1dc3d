"""Pivots of FP16/BF16 factorizations whose FP32 arrays are padded: the exported
interchanges are those of the unpadded blocks."""
import numpy as np
import pytest
import scipy.linalg as sla

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


# (points, leaf, tolerance, eta)
SIZES = [(130, 66, 1e-10, 1.0), (519, 66, 1e-6, 1.0), (1003, 64, 1e-10, 1.0), (2999, 200, 1e-4, 1.0),
         (1600, 49, 1e-10, 0.0), (3100, 97, 1e-10, 1.0)]


@pytest.mark.parametrize("n,leaf,tol,eta", SIZES)
def test_pivots_without_padding(B, n, leaf, tol, eta):
    """With the elimination in FP64, LAPACK's pivots of the exported FP32 blocks
    (root and leaves); in FP32, a valid sequence: k <= piv[k] < dimension."""
    S = B.H2Solver.build(W.cube_points(n, 3), kernel="laplace_eps", diag_shift=-999.0, leaf=leaf, eta=eta, tol=tol,
                         far_samples=512, near_samples=32)  # (a diagonal of 1: rows are exchanged)
    lv = S.stats()["levels"]
    L = len(lv) - 1
    D0, D, K, nb = lv[0]["D"], lv[L]["D"], lv[L]["K"], lv[L]["nb"]
    R = D - K
    for rr in (0, 1):
        S.set_option("rr_lu_fp64", rr)
        S.factor("fp16")
        rp, lp = S.export("root_piv", 0), S.export("piv", L).reshape(nb, R)
        assert rp.shape == (D0,)
        for p, d in [(rp, D0)] + [(q, R) for q in lp]:
            assert (np.arange(d) <= p).all() and (p < d).all()
        if rr:
            A0 = S.export("A", 0).reshape(D0, D0).astype(np.float64)
            assert (rp == sla.lu_factor(A0)[1]).all() and (rp != np.arange(D0)).any()
            Ah = S.export("Ahat", L).reshape(-1, D, D)[0][:R, :R].astype(np.float64)
            assert (lp[0] == sla.lu_factor(Ah)[1]).all()
