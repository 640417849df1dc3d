"""GPU construction at the shapes where its kernels change form: the pivoted
QR's cluster size and columns per warp (from the box dimension and the box
count), its rows per lane (from the sketch width), the column splits of the
close-field weights and the sample splits of the sketch, with ragged leaves."""
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


# leaf dimensions 12 .. 256 (one to eight columns a warp, three or five rows a
# lane), 2 to 256 boxes a level (clusters of 8 down to 1)
@pytest.mark.parametrize("n,leaf,kernel", [(90, 30, "laplace_eps"), (1500, 12, "yukawa_eps"), (3001, 64, "laplace_eps"),
                                           (2500, 100, "yukawa_eps"), (6007, 129, "laplace_eps"),
                                           (8192, 256, "yukawa_eps"), (13001, 200, "gaussian"),
                                           (25003, 128, "yukawa_eps")])
def test_construction_shapes(B, n, leaf, kernel):
    """Every basis interpolates its skeleton points (one unit row per
    skeleton), and A_H2 reproduces exact rows of A within a factor 4 of the
    plain host build (a capped randomized sketch picks somewhat worse
    skeletons than a pivoted QR of the whole composite matrix)."""
    from oracle.kernels import Kernel
    P = W.cube_points(n, 7)
    shift = {"yukawa_eps": 1.0, "gaussian": 1.0}.get(kernel, 0.0)
    kw = dict(kernel=kernel, leaf=leaf, tol=1e-8, ell=0.5, diag_shift=shift, far_samples=1024, near_samples=64)
    S = B.H2Solver.build_gpu(P, **kw)
    st = S.stats()
    assert st["construction"]["gpu_levels"] == st["L"]
    for l in range(1, st["L"] + 1):
        lv = st["levels"][l]
        X = S.export("X", l).reshape(lv["nb"], lv["D"], lv["K"])
        assert np.all(np.isfinite(X))
        unit = (X == 1.0) & (np.abs(X).sum(axis=2, keepdims=True) == 1.0)
        assert np.all(unit.sum(axis=1) >= 1)
    rows = np.random.default_rng(5).choice(n, min(n, 128), replace=False)
    x = W.uniform_rhs(n, 82)
    exact = Kernel(kernel, ell=0.5, diag_shift=shift).matrix(P, rows, np.arange(n)) @ x

    def err(solver):
        return np.linalg.norm(solver.matvec(x)[rows] - exact) / np.linalg.norm(exact)

    S0 = B.H2Solver.build(P, **kw)
    e0, eg = err(S0), err(S)
    print(f"n={n} leaf={leaf} {kernel}: sampled-row error plain {e0:.2e}, GPU {eg:.2e}")
    assert eg <= max(4.0 * e0, 1e-9)
    S0.close()
    S.close()


@pytest.mark.parametrize("n,leaf", [(3, 1), (15, 1), (21, 1)])
def test_empty_boxes(B, n, leaf):
    """More boxes than points: levels of rank 0, as the host construction has
    them (the same blocks, so products equal to the last bits)."""
    P = W.cube_points(n, 3)
    kw = dict(kernel="yukawa_eps", diag_shift=1.0, leaf=leaf, eta=1.0, tol=1e-8, far_samples=64, near_samples=8)
    G, H = B.H2Solver.build_gpu(P, **kw), B.H2Solver.build(P, **kw)
    assert [d["K"] for d in G.stats()["levels"]] == [d["K"] for d in H.stats()["levels"]]
    x = W.uniform_rhs(n, 4)
    assert np.linalg.norm(G.matvec(x) - H.matvec(x)) <= 1e-14 * np.linalg.norm(H.matvec(x))
