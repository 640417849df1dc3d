"""Instances whose leaf blocks are kept as symmetric halves while their
couplings are not: ranks that are no multiple of 4 beside leaves of a
tensor-core shape, and an imported far list that is not closed under (i, j) ->
(j, i).  The FP32 operator of the mixed refinement then takes the general form
of the couplings with the halves of the leaf blocks."""
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


def check_arithmetics(S, n):
    """FP32 sums of at most some thousand terms: 1e-6; FP32 pairs: 2^-44 (the
    bounds of the other shapes)."""
    x = W.uniform_rhs(n, 4)
    y = S.matvec(x)
    assert np.linalg.norm(S.matvec_arith(x, "fp32") - y) <= 1e-6 * np.linalg.norm(y)
    assert np.linalg.norm(S.matvec_arith(x, "fp32_pair") - y) <= 2.0 ** -44 * np.linalg.norm(y)


@pytest.mark.parametrize("n,leaf,rank", [(2048, 256, 77), (4096, 256, 98), (2048, 128, 50), (2048, 128, 33)])
def test_halves_with_odd_ranks(B, n, leaf, rank):
    S = B.H2Solver.build(W.cube_points(n, 3), kernel="yukawa_eps", diag_shift=1.0, leaf=leaf, eta=1.0, tol=1e-12,
                         max_rank=rank, far_samples=512, near_samples=32)
    lv = S.stats()["levels"]
    assert lv[-1]["D"] % 128 == 0 and lv[-1]["K"] == rank and any(d["FP"] > 0 for d in lv)
    check_arithmetics(S, n)
    b = W.uniform_rhs(n, 5)
    for prec in ("fp16", "bf16"):
        S.factor(prec)
        x, rel, _ = S.solve(b, target=1e-10, max_iters=300)
        assert rel <= 1e-10 and np.linalg.norm(b - S.matvec(x)) <= 2e-10 * np.linalg.norm(b)


@pytest.mark.parametrize("which", ["far", "near"])
@pytest.mark.parametrize("n,leaf", [(1024, 128), (1000, 66)])
def test_open_lists(B, n, leaf, which):
    """A list that holds (j, i) without (i, j) at the leaves, with and without
    padding of the FP32 arrays (leaves of 63 points)."""
    from oracle.construct import construct
    from oracle.instance import flatten
    from oracle.kernels import Kernel
    H = construct(W.cube_points(n, 3), Kernel("yukawa_eps", diag_shift=1.0), leaf, 1.0, 1e-8, 0, 256, 32)
    flat = flatten(H)
    l = max(k for k in range(flat["L"] + 1) if len(flat["far"][k]))
    pairs = flat[which][l]
    q = np.flatnonzero(pairs[:, 0] != pairs[:, 1])[-1]
    flat[which][l] = np.ascontiguousarray(np.delete(pairs, q, axis=0))
    S = B.H2Solver.from_instance(flat, kernel="yukawa_eps", leaf=leaf, eta=1.0, tol=1e-8, far_samples=256,
                                 near_samples=32, diag_shift=1.0)
    check_arithmetics(S, n)


@pytest.mark.parametrize("n,leaf,rank,precs", [(2048, 256, 232, ("fp64",)), (2048, 256, 240, ("fp64", "fp16")),
                                               (2912, 364, 332, ("fp16",))])
def test_few_complement_rows_beside_a_high_rank(B, n, leaf, rank, precs):
    """Per-box matrices of [x^R; x^S] too large for the slices that the cluster
    form of the substitution keeps in shared memory (K = 232 and above in FP64,
    332 in FP32, at 32 complement rows and fewer), against plain launches."""
    S = B.H2Solver.build(W.cube_points(n, 3), kernel="yukawa_eps", diag_shift=1.0, leaf=leaf, eta=1.0, tol=1e-14,
                         max_rank=rank, far_samples=512, near_samples=0)
    assert S.stats()["levels"][-1]["K"] == rank
    b = W.uniform_rhs(n, 5)
    for prec in precs:
        S.factor(prec)
        z = [S.ulv_apply(b)]
        S.set_option("box_stream", 2)  # (process-wide)
        try:
            z.append(S.ulv_apply(b))
        finally:
            S.set_option("box_stream", 0)
        u = 2.0 ** -53 if prec == "fp64" else 2.0 ** -24
        assert np.linalg.norm(z[0] - z[1]) <= 1e3 * u * np.linalg.norm(z[1]), prec
        x, rel, _ = S.solve(b, target=1e-10, max_iters=100)
        assert rel <= 1e-10 and np.linalg.norm(b - S.matvec(x)) <= 2e-10 * np.linalg.norm(b)


def test_tensor_core_rank_above_a_padded_level(B):
    """A rank of 128 (16-bit couplings) over a level whose rank of 125 is padded
    in the FP32 arrays: three more skeletons at level 1 of an instance whose
    ranks the construction left at 125."""
    from oracle.construct import construct
    from oracle.instance import flatten
    from oracle.kernels import Kernel
    n = 800
    H = construct(W.cube_points(n, 3), Kernel("yukawa_eps", diag_shift=1.0), 200, 0.0, 1e-13, 125, 0, 0)
    flat = flatten(H)
    assert list(flat["K"]) == [0, 125, 125] and len(flat["far"][1]) and len(flat["far"][2])
    X, SK = np.zeros((2, 250, 128)), np.zeros((2, 128), dtype=np.int64)
    for i in range(2):
        rows = np.concatenate([flat["SK"][2][2 * i], flat["SK"][2][2 * i + 1]])  # the box's points
        X[i, :, :125], SK[i, :125] = flat["X"][1][i], flat["SK"][1][i]
        more = np.flatnonzero(~np.isin(rows, SK[i, :125]))[:3]
        X[i, more, :] = 0.0
        X[i, more, 125 + np.arange(3)] = 1.0
        SK[i, 125:] = rows[more]
    flat["X"][1], flat["SK"][1] = X, SK
    flat["K"] = np.array([0, 128, 125], dtype=np.int32)
    flat["D"] = np.array([256, 250, 200], dtype=np.int32)
    S = B.H2Solver.from_instance(flat, kernel="yukawa_eps", leaf=200, eta=0.0, tol=1e-13, max_rank=128, far_samples=0,
                                 near_samples=0, diag_shift=1.0)
    check_arithmetics(S, n)
    S.factor("fp64")
    sh64 = S.export("Shat", 2)
    b = W.uniform_rhs(n, 5)
    for prec in ("fp16", "bf16"):
        S.factor(prec)
        # (T in FP32 is within 1e-3 of the FP64 one; it stands on both sides)
        sh = S.export("Shat", 2).astype(np.float64)
        assert sh.shape == sh64.shape
        assert np.linalg.norm(sh - sh64) <= 2e-3 * np.linalg.norm(sh64)
        x, rel, _ = S.solve(b, target=1e-10, max_iters=100)
        assert rel <= 1e-10 and np.linalg.norm(b - S.matvec(x)) <= 2e-10 * np.linalg.norm(b)


@pytest.mark.parametrize("n,leaf", [(130, 33), (1000, 128)])
def test_rank_zero(B, n, leaf):
    """An imported instance of rank 0 on every level: boxes of dimension 0 above
    the leaves, and the near blocks alone (products against the blocks)."""
    from oracle.construct import construct
    from oracle.instance import flatten
    from oracle.kernels import Kernel
    flat = flatten(construct(W.cube_points(n, 3), Kernel("yukawa_eps", diag_shift=1.0), leaf, 1.0, 1e-6, 0, 64, 8))
    L, D = flat["L"], int(flat["D"][-1])
    flat["K"] = np.zeros(L + 1, dtype=np.int32)
    flat["D"] = np.array([0] * L + [D], dtype=np.int32)
    flat["far"] = [np.zeros((0, 2), dtype=np.int32) for _ in range(L + 1)]
    flat["X"] = [None] + [np.zeros((2 ** l, flat["D"][l], 0)) for l in range(1, L + 1)]
    flat["SK"] = [None] + [np.zeros((2 ** l, 0), dtype=np.int64) for l in range(1, L + 1)]
    S = B.H2Solver.from_instance(flat, kernel="yukawa_eps", leaf=leaf, eta=1.0, tol=1e-6, far_samples=64,
                                 near_samples=8, diag_shift=1.0)
    A = S.export("A", L).reshape(-1, D, D)
    off, perm = flat["leaf_offsets"], flat["perm"]
    x = W.uniform_rhs(n, 4)
    y = np.zeros(n)
    for q, (i, j) in enumerate(flat["near"][L]):
        pi, pj = perm[off[i]:off[i + 1]], perm[off[j]:off[j + 1]]
        y[pi] += A[q][:len(pi), :len(pj)] @ x[pj]
    assert np.linalg.norm(S.matvec(x) - y) <= 1e-13 * np.linalg.norm(y)
    check_arithmetics(S, n)
    for prec in ("fp64", "fp16"):
        S.factor(prec)
        xs, rel, _ = S.solve(x, target=1e-10, max_iters=200)
        assert rel <= 1e-10 and np.linalg.norm(x - S.matvec(xs)) <= 2e-10 * np.linalg.norm(x)
