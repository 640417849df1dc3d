"""FP16/BF16 factorizations whose box dimensions or ranks are no multiples of
4: the FP32 arrays are padded, what the library returns is not.  Sizes around
the padding's edges: odd and even leaves and ranks, ranks that differ between
levels (tolerance ranks), one level, leaves that need no padding."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

U32 = 2.0 ** -24


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
         (1600, 49, 1e-10, 0.0), (3100, 97, 1e-10, 1.0), (4011, 255, 1e-10, 1.0)]


@pytest.mark.parametrize("n,leaf,tol,eta", SIZES)
def test_padded_levels_against_fp64_products(B, n, leaf, tol, eta):
    """FP32 and FP32-pair matvecs against the FP64 one, the projected blocks
    against U_i^T A_ij U_j in FP64 from the exported FP32 bases (a D-term sum
    in FP32, twice: 4 D u32 of the block's norm), the bases' orthogonality
    (1e-5, the bound of the unpadded shapes), and the refined solution."""
    P = W.cube_points(n, 3)
    S = B.H2Solver.build(P, kernel="yukawa_eps", diag_shift=1.0, leaf=leaf, eta=eta, tol=tol, far_samples=512,
                         near_samples=32)
    st = S.stats()
    L = st["L"]
    x = W.uniform_rhs(n, 4)
    y = S.matvec(x)
    assert np.linalg.norm(S.matvec_arith(x, "fp32") - y) <= 1e-6 * np.linalg.norm(y)
    assert np.linalg.norm(S.matvec_arith(x, "fp32_pair") - y) <= 2.0 ** -44 * np.linalg.norm(y)
    S.factor("fp16")
    lv = st["levels"][L]
    nb, D, K = lv["nb"], lv["D"], lv["K"]
    U = S.export("U", L).reshape(nb, D, D).astype(np.float64)
    for i in range(nb):
        assert np.abs(U[i] @ U[i].T - np.eye(D)).max() <= 1e-5
    # the diagonal pair of box 0 is the list's first: all of it but SS, which
    # holds the Schur update
    A = S.export("A", L).reshape(-1, D, D)
    Ah = S.export("Ahat", L).reshape(-1, D, D).astype(np.float64)
    ref = U[0] @ A[0] @ U[0].T
    R = D - K
    got = Ah[0].copy()
    got[R:, R:] = ref[R:, R:]
    tc = st["levels"][L]["D"] % 128 == 0
    assert np.linalg.norm(got - ref) <= (4e-3 if tc else 4 * D * U32) * np.linalg.norm(ref)
    inv = S.export("Ainv", L).reshape(nb, R, R).astype(np.float64)
    full = Ah[0][:R, :R]
    assert np.linalg.norm(inv[0] @ full - np.eye(R)) <= 1e-4 * R
    assert S.export("T", L).size == nb * K * K and S.export("Shat", L).size in (lv["FP"] * K * K,)
    D0 = st["levels"][0]["D"]
    A0 = S.export("A", 0).reshape(D0, D0).astype(np.float64)
    inv0 = S.export("root_inv", 0).reshape(D0, D0).astype(np.float64)
    assert np.linalg.norm(inv0 @ A0 - np.eye(D0)) <= 1e-4 * D0
    assert sorted(set(S.export("root_piv", 0))) <= list(range(D0))
    b = W.uniform_rhs(n, 5)
    for prec in ("fp16", "bf16"):
        S.factor(prec)
        xs, rel, _ = S.solve(b, target=1e-11, max_iters=200)
        assert rel <= 1e-11 and np.linalg.norm(b - S.matvec(xs)) <= 2e-11 * np.linalg.norm(b)
    z = S.ulv_apply(b)
    S.factor("fp64")
    z64 = S.ulv_apply(b)
    assert np.linalg.norm(z - z64) <= (8e-2 if tc else 1e-3) * np.linalg.norm(z64)
    x64, _, _ = S.solve(b, target=1e-11, max_iters=200)
    assert np.linalg.norm(x64 - xs) <= 1e-9 * np.linalg.norm(x64)
    S.close()
