"""The work that programs have this library do, as timed cases.

A case is one call sequence through the package's public entry points on a problem of the
repository's own kind: -div(nu grad u) = f on a Cartesian grid, discretised with SIPG blocks,
the coefficient jumping across a ball or log-normal per cell, right-hand sides iid U[-1, 1].

Kinds of case:
  solve         KCycleSolver.solve / kcmg_solve with a budget of level-0 cycles (``cycles``), or
                to a tolerance (``rtol``).  Budgets are how a program uses the solver inside an
                outer loop; they also keep the iterates of different builds comparable.
  adjoint       kcmg_solve_adjoint and kcmg_grad_lognu: the backward pass of autograd.KCycleSolve
  solve_multi   one solve of several right-hand sides
  apply         y = A x on the finest level
  residual      r = b - A x and its norm without any allocation (error-recovery path)
  smooth        one smoother call on the finest level
  smooth_multi  the same for several right-hand sides
"""
from __future__ import annotations

import functools
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2512_08728_gb300 as pkg
from workloads import neighbours, prolongation_matrices, reference_matrices
from workloads.sipg import centroids

DEV = "cuda"


def listed():
    case = _case
    return [
        # the smallest solve of the tests and of smoke(): every launch and round trip counts
        case("solve_2d_p1_16x16", "solve", 2, 1, (16, 16), 3, rtol=1e-11),
        # a mixed-precision solve to tolerance: FP32 sweeps under FP64 minimisation
        case("solve_3d_p2_8cube_mixed", "solve", 3, 2, (8, 8, 8), 3, precision="mixed", rtol=1e-11),
        # a 2-D Poisson problem of the paper's size and degree range, the task-parallel cycle
        case("solve_2d_p3_128x96", "solve", 2, 3, (128, 96), 5, m=8, lmax=200, cycles=2),
        # the benchmark's workload in its timed configuration, bounded to a few cycles
        case("solve_3d_p2_64cube", "solve", 3, 2, (64, 64, 64), 5, m=12, lmax=400, cycles=5),
        # the stretched high-contrast p = 3 problem, which needs the Schwarz smoother
        case("solve_3d_p3_24cube_schwarz", "solve", 3, 3, (24, 24, 24), 4, m=12, lmax=400, cycles=1,
             lz=10.0, inside=1.0e4, smoother="as", omega=0.5, sweeps=2),
        # the backward pass of the coefficient-gradient workload
        case("adjoint_3d_p2_32cube", "adjoint", 3, 2, (32, 32, 32), 4, nu="lognormal", lmax=200, cycles=2),
        # a few right-hand sides on a small grid, to tolerance: launches and host control
        case("multi_3d_p2_8cube_rhs8", "solve_multi", 3, 2, (8, 8, 8), 3, nrhs=8, rtol=1e-11),
        # the full batch width on the batched workload's grid
        case("multi_3d_p2_32cube_rhs32", "solve_multi", 3, 2, (32, 32, 32), 4, nrhs=32, m=12, lmax=100, cycles=1),
        # single operations at the sizes of the benchmark and of the larger configurations
        case("apply_3d_p2_64cube", "apply", 3, 2, (64, 64, 64), 5),
        case("residual_3d_p1_96x80x72", "residual", 3, 1, (96, 80, 72), 4),
        case("smooth_3d_p2_64cube_bf16", "smooth", 3, 2, (64, 64, 64), 5, precision="mixed_bf16"),
        case("smooth_multi_3d_p2_48cube_rhs32", "smooth_multi", 3, 2, (48, 48, 48), 4, nrhs=32,
             precision="mixed_bf16"),
    ]


def _case(name, kind, d, p, n, levels, nu="jump", inside=1000.0, lz=1.0, precision="fp64", m=0, lmax=0,
          cycles=0, rtol=1e-10, smoother="bj", omega=0.7, sweeps=5, nrhs=1):
    n = tuple(n) + (1,) * (3 - len(n))
    return {"name": name, "kind": kind, "d": d, "p": p, "nx": n[0], "ny": n[1], "nz": n[2], "levels": levels,
            "nu": nu, "inside": inside, "lz": lz, "precision": precision, "m": m, "lmax": lmax,
            "cycles": cycles, "rtol": rtol, "smoother": smoother, "omega": omega, "sweeps": sweeps,
            "nrhs": nrhs}


# ------------------------------------------------------------------ drawn cases
def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "adjoint", "solve_multi", "apply", "residual", "smooth",
                       "smooth_multi"])
    kw, nrhs = {}, 1
    d, p = rng.choice([(2, 1), (2, 2), (2, 3), (3, 1), (3, 2), (3, 2), (3, 2), (3, 3)])
    top = 2.6e6                                     # unknowns of the largest listed operator
    small = {2: 2.0e3, 3: 5.2e3}                    # unknowns of the solves run to tolerance
    if kind == "solve":
        form = rng.choice(["multiplicative", "task-parallel", "task-parallel", "schwarz", "to tolerance"])
        if form == "to tolerance":
            d, p = rng.choice([(2, 1), (2, 2), (3, 1), (3, 2)])
            kw, top = dict(precision=rng.choice(["fp64", "mixed", "mixed_bf16"]), rtol=1e-11), small[d]
        elif form == "schwarz":
            kw, top = dict(m=rng.choice([4, 8, 12]), lmax=rng.choice([200, 400]), cycles=1, smoother="as",
                           omega=0.5, sweeps=2, lz=rng.choice([1.0, 10.0])), 3e5
        else:
            kw = dict(m=0 if form == "multiplicative" else rng.choice([4, 8, 12]), lmax=rng.choice([100, 200, 400]),
                      cycles=rng.choice([1, 1, 2]))
    elif kind == "adjoint":
        d, p = rng.choice([(2, 2), (3, 1), (3, 2), (3, 2)])
        kw, top = dict(nu="lognormal", lmax=200, cycles=rng.choice([1, 2])), 4e5
    elif kind == "solve_multi":
        nrhs = rng.choice([3, 5, 8, 12, 17, 24, 32])
        if rng.random() < 0.4:
            d, p = rng.choice([(2, 1), (3, 1), (3, 2)])
            kw, top = dict(rtol=1e-11), small[d]
        else:
            if nrhs > 12:
                p = 1
            kw, top = dict(nu="lognormal", m=rng.choice([0, 0, 8]), lmax=100, cycles=1), 7e6 / nrhs
    elif kind == "smooth":
        kw = dict(precision=rng.choice(["fp64", "mixed", "mixed_bf16"]))
    elif kind == "smooth_multi":
        d, p, nrhs = 3, 2, 32
        kw, top = dict(precision=rng.choice(["mixed", "mixed_bf16"])), 1.1e6
    if "nu" not in kw and rng.random() < 0.3:
        kw["nu"] = "lognormal"
    np_ = math.comb(p + d, d)
    low = 2.0e5 if kind == "smooth_multi" else 700.0
    cells = math.exp(rng.uniform(math.log(low / np_), math.log(top / np_)))
    # the coarsest level, solved directly, is left with 2-4 (3-D) or 4-8 (2-D) cells a side (a
    # single smoother call needs no deep hierarchy)
    side = cells ** (1.0 / d)
    levels = 2
    deepest = 4 if kind == "smooth_multi" else 5 if d == 3 else 7
    while levels < deepest and side / 2 ** levels >= (2.0 if d == 3 else 4.0):
        levels += 1
    unit = 2 ** (levels - 1)
    n = [max(1, round(side * f / unit)) * unit for f in (rng.uniform(0.75, 1.0), rng.uniform(0.85, 1.0), 1.0)[:d]]
    c = _case("", kind, d, p, n, levels, nrhs=nrhs, **kw)
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs
def _problem(c, seed):
    """Operator blocks, hierarchy and right-hand side of a case on the GPU (the arithmetic of
    workloads.sipg.assemble, so that a symmetric operator is stored bitwise symmetric)."""
    d, p = c["d"], c["p"]
    n = (c["nx"], c["ny"], c["nz"])[:d]
    h = np.ones(d) / np.array(n)
    h[-1] *= c["lz"]
    rng = np.random.default_rng(seed)
    ref = reference_matrices(d, p, h, 4.0 * (p + 1) ** 2)
    mid = centroids(n, 1.0 / np.array(n, dtype=np.float64))
    inside = np.sum((mid - 0.5) ** 2, axis=1) < 0.3 ** 2
    if c["nu"] == "jump":
        nu = np.where(inside, c["inside"], 1.0)
    else:
        nu = np.exp(rng.standard_normal(mid.shape[0]) + np.where(inside, math.log(c["inside"]), 0.0))
    nbr = torch.from_numpy(neighbours(n)).to(DEV).long()
    v = torch.from_numpy(nu).to(DEV)
    V, F, B = (torch.from_numpy(ref[k]).to(DEV) for k in "VFB")
    np_ = V.shape[0]
    blocks = torch.zeros(2 * d + 1, v.numel(), np_, np_, dtype=torch.float64, device=DEV)
    col = lambda t: t[:, None, None]  # noqa: E731
    blocks[0] = col(v) * V
    for k in range(d):
        g, has = [], []
        for side in (0, 1):
            J = nbr[:, 2 * k + side]
            has.append(J >= 0)
            o = v[J.clamp(min=0)]
            g.append(torch.where(has[-1], 2.0 * (v * o) / (v + o), torch.zeros_like(v)))
        zero = torch.zeros_like(v)
        blocks[0] += (col(g[1]) * F[k, 0] + col(torch.where(has[1], zero, v)) * B[k, 1]
                      + col(g[0]) * F[k, 3] + col(torch.where(has[0], zero, v)) * B[k, 0])
        blocks[1 + 2 * k] = col(g[0]) * F[k, 2]
        blocks[2 + 2 * k] = col(g[1]) * F[k, 1]
    N = v.numel() * np_
    gen = torch.Generator(device=DEV).manual_seed(int(seed) % (1 << 62))
    shape = (N,) if c["nrhs"] == 1 else (N, c["nrhs"])
    rand = lambda s: torch.rand(s, dtype=torch.float64, device=DEV, generator=gen) * 2.0 - 1.0  # noqa: E731
    pr = SimpleNamespace(d=d, np_=np_, n=n, nlevels=c["levels"], ndof=N, blocks=blocks, nbr=nbr,
                         prolong=prolongation_matrices(d, p), ref=ref, nu=nu, b=rand(shape))
    pr.x = rand(shape)
    return pr


def prepare(case, seed):
    """The context of the operator (a program keeps it), the inputs on the device, and the
    stream the program works on."""
    c = case
    pr = _problem(c, seed)
    torch.cuda.synchronize()
    stream = torch.cuda.Stream()
    solver = pkg.KCycleSolver(pr, precision=c["precision"], lmax=c["lmax"], async_smooth=c["m"],
                              smoother=c["smoother"], omega=c["omega"], sweeps=c["sweeps"],
                              stream=stream.cuda_stream)
    st = SimpleNamespace(case=c, solver=solver, stream=stream, b=pr.b, x=pr.x)
    if c["kind"] == "adjoint":   # field, reference matrices and forward solution of the backward pass
        dev = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).to(DEV)  # noqa: E731
        st.nu, st.ref = dev(pr.nu), {k: dev(pr.ref[k]) for k in "VFB"}
    if c["kind"] == "residual":
        st.r = torch.empty_like(pr.b)
    torch.cuda.synchronize()
    return st


# ------------------------------------------------------------------ one pass
def run(st):
    c, s = st.case, st.solver
    kind = c["kind"]
    with torch.cuda.stream(st.stream):
        if kind in ("solve", "solve_multi"):
            x, info = s.solve(st.b, rtol=c["rtol"], maxiter=c["cycles"] or 300)
            return {"x": x}
        if kind == "adjoint":
            lam, info = s.solve(st.b, rtol=c["rtol"], maxiter=c["cycles"], adjoint=True)
            return {"lambda": lam, "g": s.grad_lognu(st.nu, st.ref, lam, st.x)}
        if kind == "apply":
            return {"y": s.apply(0, st.x)}
        if kind == "residual":
            return {"norm": pkg.kcmg_residual_noalloc(s.ctx, st.b, st.x, st.r), "r": st.r}
        if kind == "smooth":
            return {"z": s.smooth(0, st.b)}
        return {"z": s.smooth_multi(0, st.b)}


# ------------------------------------------------------------------ what a pass needs at least
@functools.lru_cache(maxsize=None)
def _nonzeros(d, p):
    """Entries of a cell's coupling blocks and of its diagonal block that are not zero."""
    ref = reference_matrices(d, p, np.ones(d), 4.0 * (p + 1) ** 2)
    off = sum(int(np.count_nonzero(ref["F"][k, j])) for k in range(d) for j in (1, 2))
    diag = ref["V"] != 0
    for k in range(d):
        diag = diag | (ref["F"][k, 0] != 0) | (ref["F"][k, 3] != 0)
    return off, int(np.count_nonzero(diag))


def work(case):
    """The operator's nonzero entries and the vectors read once, results written once; the
    multiplications and additions of the finest level (the coarse levels add to a solve)."""
    c = case
    off, diag = _nonzeros(c["d"], c["p"])
    np_ = math.comb(c["p"] + c["d"], c["d"])
    cells, R = c["nx"] * c["ny"] * c["nz"], c["nrhs"]
    N = cells * np_ * R
    es = 8 if c["precision"] == "fp64" else 4
    ei = {"fp64": 8, "mixed": 4}.get(c["precision"], 2)
    if c["smoother"] == "as":
        mat = 2 * np_ * np_ * 2 ** c["d"]                      # two patch inverses per cell
        sweep, first = off + diag + mat, mat
    else:
        sweep, first = off + np_ * np_, np_ * np_
        mat = np_ * np_
    smooth = 2.0 * cells * R * (first + (c["sweeps"] - 1) * sweep)
    spmv = 2.0 * cells * R * (off + diag)
    kind = c["kind"]
    if kind == "apply":
        return {"bytes": 8.0 * (cells * (off + diag) + 2 * N), "flops": spmv}
    if kind == "residual":
        return {"bytes": 8.0 * (cells * (off + diag) + 3 * N), "flops": spmv + 3.0 * N}
    if kind in ("smooth", "smooth_multi"):
        return {"bytes": float(cells) * (off * es + mat * ei) + 16.0 * N, "flops": smooth}
    cycles = c["cycles"] or 30
    calls, rms = (c["m"], c["m"] + 1) if c["m"] else (2, 3)
    l = cycles * rms
    flops = cycles * (calls * smooth + rms * spmv) + 3.0 * l * (l - 1) * N
    return {"bytes": cells * 8.0 * (off + diag) + cells * (off * es + mat * ei) + 24.0 * N, "flops": flops}


# ------------------------------------------------------------------ the same in plain torch, 64 bits
def _apply(pr, x):
    n = pr.np_
    X = x.reshape(pr.nbr.shape[0], n, -1)
    y = torch.einsum("cij,cjr->cir", pr.blocks[0], X)
    for s in range(1, pr.blocks.shape[0]):
        J = pr.nbr[:, s - 1]
        y += torch.einsum("cij,cjr->cir", pr.blocks[s], X[J.clamp(min=0)] * (J >= 0)[:, None, None])
    return y.reshape(x.shape)


def _smooth(c, pr, r):
    C, n = pr.nbr.shape[0], pr.np_
    D = pr.blocks[0].reshape(C, n, n)
    off = SimpleNamespace(np_=n, nbr=pr.nbr, blocks=pr.blocks.clone())
    off.blocks[0] = 0.0
    inv = torch.linalg.inv(D)
    z = torch.zeros_like(r)
    for k in range(c["sweeps"]):
        t = r - _apply(off, z) if k else r
        e = torch.einsum("cij,cjr->cir", inv, t.reshape(C, n, -1)).reshape(r.shape)
        z = (1.0 - c["omega"]) * z + c["omega"] * e
    return z


def _solution(pr):
    C, n = pr.nbr.shape[0], pr.np_
    A = torch.zeros(C, n, C, n, dtype=torch.float64, device=DEV)
    K = torch.arange(C, device=DEV)
    A[K, :, K, :] = pr.blocks[0]
    for s in range(1, pr.blocks.shape[0]):
        J = pr.nbr[:, s - 1]
        ok = J >= 0
        A[K[ok], :, J[ok], :] = pr.blocks[s][ok]
    A = A.reshape(C * n, C * n)
    return torch.linalg.solve(A, pr.b)


def exact(case, seed):
    c = case
    kind = c["kind"]
    if kind in ("solve", "solve_multi", "adjoint") and c["cycles"]:
        return None          # an unfinished iterate has no value of its own
    pr = _problem(c, seed)
    if kind in ("solve", "solve_multi"):
        return {"x": _solution(pr)}
    if kind == "apply":
        return {"y": _apply(pr, pr.x)}
    if kind == "residual":
        r = pr.b - _apply(pr, pr.x)
        return {"norm": float(torch.linalg.vector_norm(r)), "r": r}
    return {"z": _smooth(c, pr, pr.b)}
