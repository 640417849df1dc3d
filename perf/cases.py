"""The calls that users of the H^2-ULV solver spend their time in, as cases
to be measured: factor and solve over the range of sizes, point sets, kernels
and precisions, solves with a factorization that is kept, matvecs, a batch of
uneven systems, and the construction from new points.

A case is a dict of plain values:
  op       "step"   factor, then one refined solve to 1e-10 (new matrix entries
                    or a new precision on a structure that is kept)
           "solve"  refined solves of nrhs right-hand sides with a
                    factorization that is kept
           "matvec" y = A_H2 x in FP64 for nrhs vectors
           "forest" a batch of uneven systems, factor and solve of all
           "build"  construction on the GPU from new points, and one matvec
  n        points (a forest: of its largest system)
  geometry "cube" (uniform in the unit cube) or "sphere" (on its surface)
  kernel   "yukawa_eps" (+ 1 on the diagonal), "laplace_eps" or "gaussian"
  leaf, tol, prec, nrhs, systems
"""
import math
import random

import numpy as np
import torch

from paper_2502_02395_gb300.binding import H2Batch, H2Solver

TARGET = 1e-10
MAX_ITERS = 300
EPS = 1e-3


def _case(op, n, geometry="cube", kernel="yukawa_eps", leaf=256, tol=1e-10, prec="fp16", nrhs=1, systems=1):
    return dict(op=op, n=n, geometry=geometry, kernel=kernel, leaf=leaf, tol=tol, prec=prec, nrhs=nrhs,
                systems=systems)


def listed():
    return [
        # the smallest system in use: the size of the first solver workload
        dict(name="step_cube2048", **_case("step", 2048, kernel="laplace_eps", leaf=64)),
        # a few thousand points, a count that fills no power of two, BF16
        dict(name="step_cube6007_bf16", **_case("step", 6007, leaf=128, tol=1e-8, prec="bf16")),
        # the medium volume problem, full leaves
        dict(name="step_cube32768", **_case("step", 32768)),
        # the usual case in practice: a point count that fills no leaf (196 of 256)
        dict(name="step_cube50021", **_case("step", 50021)),
        # points on a surface, whose boxes have a third of the neighbours
        dict(name="step_sphere65536", **_case("step", 65536, geometry="sphere", kernel="laplace_eps", tol=1e-8)),
        # the headline workload
        dict(name="step_cube262144", **_case("step", 262144)),
        # double precision throughout
        dict(name="step_sphere8192_fp64",
             **_case("step", 8192, geometry="sphere", kernel="laplace_eps", tol=1e-8, prec="fp64")),
        # several right-hand sides against a factorization that is kept
        dict(name="solve_cube16384_x4", **_case("solve", 16384, nrhs=4)),
        # the operator alone: one small product, and several of a large one
        dict(name="matvec_sphere3001", **_case("matvec", 3001, geometry="sphere", kernel="laplace_eps", leaf=128,
                                               tol=1e-8, prec="fp64")),
        dict(name="matvec_cube65536_x4", **_case("matvec", 65536, prec="fp64", nrhs=4)),
        # independent Gaussian-covariance systems of uneven size
        dict(name="forest_gauss6_5000", **_case("forest", 5000, kernel="gaussian", leaf=128, tol=1e-8, systems=6)),
        # new points: structure, bases and blocks from nothing
        dict(name="build_cube16384", **_case("build", 16384)),
    ]


def draw(rng):
    op = rng.choice(["step"] * 6 + ["solve", "solve", "matvec", "matvec", "forest", "build"])
    geometry = rng.choice(["cube", "cube", "sphere"])
    kernel = rng.choice(["yukawa_eps", "laplace_eps"])
    prec = rng.choice(["fp16", "fp16", "fp16", "bf16", "fp64"]) if op in ("step", "solve") else "fp16"
    tol = rng.choice([1e-8, 1e-10])
    lo, hi = {"step": (2048, 131072), "solve": (2048, 49152), "matvec": (2048, 131072), "forest": (4096, 6000),
              "build": (4096, 32768)}[op]
    if prec == "fp64":
        hi = 12000
    n = int(math.exp(rng.uniform(math.log(lo), math.log(hi))))
    nrhs = rng.choice([1, 2, 3, 4]) if op in ("solve", "matvec") else 1
    if op == "forest":
        return _case(op, n, kernel="gaussian", leaf=128, tol=1e-8, systems=rng.choice([3, 4, 5, 6]))
    leaf = 64 if n < 4096 else (128 if n < 8192 else rng.choice([128, 256, 256]) if n < 16384 else 256)
    return _case(op, n, geometry, kernel, leaf, tol, "fp64" if op == "matvec" else prec, nrhs)


# ----------------------------------------------------------------- inputs ---
def _points(geometry, n, rng):
    if geometry == "cube":
        return rng.random((n, 3))
    g = rng.standard_normal((n, 3))
    return g / np.linalg.norm(g, axis=1, keepdims=True)


def _params(case):
    kw = dict(kernel=case["kernel"], leaf=case["leaf"], eta=1.0, tol=case["tol"], eps=EPS)
    if case["kernel"] == "yukawa_eps":
        kw["diag_shift"] = 1.0
    return kw


def _inputs(case, seed):
    """Points and vectors (host) of a case that is no forest."""
    rng = np.random.default_rng(seed)
    P = _points(case["geometry"], case["n"], rng)
    return P, rng.uniform(-1.0, 1.0, (case["nrhs"], case["n"]))


def _forest_inputs(case, seed):
    """Uneven systems: points over their length scales (so that one kernel
    exp(-r^2) serves all), and their right-hand sides."""
    rng = np.random.default_rng(seed)
    r = random.Random(case["n"] * 31 + case["systems"])
    ns = [case["n"]] + [int(case["n"] * r.uniform(0.83, 1.0)) for _ in range(case["systems"] - 1)]
    P = [rng.random((n, 3)) / rng.uniform(0.05, 0.5) for n in ns]
    return P, [rng.uniform(-1.0, 1.0, n) for n in ns]


def prepare(case, seed):
    if case["op"] == "forest":
        P, b = _forest_inputs(case, seed)
        kw = dict(kernel="gaussian", ell=1.0, diag_shift=1.0, leaf=case["leaf"], eta=1.0, tol=case["tol"],
                  near_samples=0)
        return dict(op="forest", batch=H2Batch.forest(P, **kw), b=b, prec=case["prec"])
    P, V = _inputs(case, seed)
    if case["op"] == "build":
        return dict(op="build", points=P, kw=_params(case), x=torch.from_numpy(V[0]).cuda())
    S = H2Solver.build_gpu(P, **_params(case))
    v = torch.from_numpy(V).cuda()
    if case["op"] == "solve":
        S.factor(case["prec"])
    return dict(op=case["op"], solver=S, v=v[0].clone() if case["op"] == "step" else v, prec=case["prec"])


def run(state):
    op = state["op"]
    if op == "step":
        state["solver"].factor(state["prec"])
        x, _, _ = state["solver"].solve(state["v"], target=TARGET, max_iters=MAX_ITERS)
        return x
    if op == "solve":
        X, _, _ = state["solver"].solve_many(state["v"], target=TARGET, max_iters=MAX_ITERS)
        return X
    if op == "matvec":
        if state["v"].shape[0] == 1:
            return state["solver"].matvec(state["v"][0])
        return state["solver"].matvec_many(state["v"])
    if op == "forest":
        X, _, _, _ = state["batch"].run(state["prec"], B=state["b"], target=TARGET, max_iters=MAX_ITERS)
        return X
    S = H2Solver.build_gpu(state["points"], **state["kw"])
    y = S.matvec(state["x"])
    S.close()
    return y


# ------------------------------------------------------------------- work ---
def _system_work(case, n):
    """(entries of the near blocks, couplings and bases, factorization flops)
    of one system: with 2^L boxes a level, about 24 near and 16 far boxes per
    box in a volume and 8.3 and 8 on a surface, blocks of D points and K = D / 2
    skeletons; of symmetric blocks one half is needed."""
    L = 0
    while case["leaf"] * 2 ** L < n:
        L += 1
    near, far = (24.0, 16.0) if case["geometry"] == "cube" else (8.3, 8.0)
    D = math.ceil(n / 2 ** L)
    K = D // 2
    entries, flops = 0.0, 0.0
    for lv in range(L, 0, -1):
        nb = 2.0 ** lv
        d = D if lv == L else 2 * K
        np_up = nb * (min(near, nb) + 1) / 2
        fp_up = nb * max(0.0, min(far, nb - near)) / 2
        if lv == L:
            entries += np_up * d * d
        entries += fp_up * K * K + nb * d * K
        # two-sided projections, couplings, QR and inverse, Schur update
        flops += np_up * 4.0 * d ** 3 + fp_up * 4.0 * K ** 3 + nb * (2.0 * d * K * K + 2.0 * (d - K) ** 3)
    return entries, flops


def work(case):
    n, r = case["n"], case["nrhs"]
    entries, flops = _system_work(case, n)
    if case["op"] == "matvec":
        # every entry of the symmetric halves read once in FP64, used twice
        return {"bytes": 8.0 * entries + 16.0 * n * r, "flops": 4.0 * entries * r}
    if case["op"] == "solve":
        return {"bytes": 8.0 * entries + 16.0 * n * r, "flops": 8.0 * entries * r}
    if case["op"] == "build":
        # the entries are made from the points and written once
        return {"bytes": 8.0 * entries + 24.0 * n + 16.0 * n, "flops": 10.0 * entries}
    s = case["systems"]
    return {"bytes": s * (8.0 * entries + 16.0 * n), "flops": s * (flops + 8.0 * entries)}


# ------------------------------------------------------------------ exact ---
def _kernel_rows(case, P, rows, scale=1.0):
    """Rows of the dense kernel matrix in FP64 (P: N x 3 on the GPU)."""
    X, Y = P[rows], P
    r2 = ((X[:, None, :] - Y[None, :, :]) ** 2).sum(-1)
    if case["kernel"] == "gaussian":
        A, diag = torch.exp(-r2), 2.0
    else:
        r = r2.sqrt()
        A = 1.0 / (r + EPS)
        diag = 1.0 / EPS
        if case["kernel"] == "yukawa_eps":
            A, diag = A * torch.exp(-r), diag + 1.0
    A[torch.arange(len(rows), device=P.device), rows] = diag
    return A


def _dense(case, P):
    P = torch.from_numpy(P).cuda()
    n = len(P)
    return torch.cat([_kernel_rows(case, P, torch.arange(i, min(i + 2048, n), device=P.device))
                      for i in range(0, n, 2048)])


def exact(case, seed):
    """The answers for the dense kernel matrix itself, which A_H2 stands for:
    products at any size here, solutions where a dense LU is quick."""
    if case["op"] == "forest":
        P, b = _forest_inputs(case, seed)
        return [torch.linalg.solve(_dense(case, p), torch.from_numpy(v).cuda()) for p, v in zip(P, b)]
    P, V = _inputs(case, seed)
    v = torch.from_numpy(V).cuda()
    if case["op"] in ("matvec", "build"):
        Pd = torch.from_numpy(P).cuda()
        y = torch.cat([_kernel_rows(case, Pd, torch.arange(i, min(i + 2048, len(P)), device=Pd.device)) @ v.T
                       for i in range(0, len(P), 2048)]).T.contiguous()
        return y[0] if case["op"] == "build" or case["nrhs"] == 1 else y
    if case["n"] > 17000:
        return None
    x = torch.linalg.solve(_dense(case, P), v.T).T.contiguous()
    return x[0] if case["op"] == "step" else x
