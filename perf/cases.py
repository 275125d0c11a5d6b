"""Performance cases: what a program that uses this library has it do, through
the binding's public calls -- preconditioner applies, SpMV, Gram-Schmidt
projections, whole Krylov solves, batched solves and numeric refactorisation
-- from one small latency-bound system to the 128^3 ones that fill the GPU.

A case is a dict of plain values; ``prepare`` makes a system from the seed
(matrix values, right-hand sides) and the handles that a program keeps;
``run`` is one pass.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1606_00545_gb300 import hecgpu as H
from paper_1606_00545_gb300 import synth


def listed():
    return [
        # M^-1 r of one small system inside a latency-bound loop: 2D, one ILU(0) block
        {"name": "apply_2d_small", "kind": "apply", "grid": "2d5", "side": 64, "k": 0, "blocks": 1,
         "f32": False},
        # M^-1 r of the headline system, FP64: 3D 7-point, ILU(1) on 64 RAS blocks
        {"name": "apply_3d_large", "kind": "apply", "grid": "3d7", "side": 128, "k": 1, "blocks": 64,
         "f32": False},
        # M^-1 r of the mixed-precision inner solves on irregular 27-point rows
        # (long rows: the generic factor layout)
        {"name": "apply_27pt_f32", "kind": "apply", "grid": "3d27i", "side": 72, "k": 0,
         "blocks": 64, "f32": True},
        # SpMV with both fused dots, as every Krylov step runs it
        {"name": "spmv_3d_large", "kind": "spmv", "grid": "3d7", "side": 128, "f32": False},
        # FP32 SpMV with a CSR tail and gathers out of order, odd size
        {"name": "spmv_27pt_f32", "kind": "spmv", "grid": "3d27i", "side": 95, "f32": True},
        # Arnoldi projection h = V^T w at the last step of a GMRES(30) cycle
        {"name": "projection", "kind": "projection", "n": 2097152, "k": 30},
        # a small system solved to convergence: every launch counts
        {"name": "gmres_2d_small", "kind": "gmres", "grid": "2d5", "side": 64, "k": 0, "blocks": 1,
         "mixed": False, "steps": 130},
        # the headline solver on the headline system, a budget of passes as a
        # time-stepping code gives it
        {"name": "bicgstab_3d_large", "kind": "bicgstab", "grid": "3d7", "side": 128, "k": 1,
         "blocks": 64, "passes": 16},
        # mixed-precision GMRES(30) to convergence on irregular 27-point rows
        {"name": "gmres_mixed_27pt", "kind": "gmres", "grid": "3d27i", "side": 64, "k": 0,
         "blocks": 64, "mixed": True, "steps": 28},
        # CG with damped Jacobi on a mid-size SPD system of odd side
        {"name": "cg_jacobi_3d", "kind": "cg", "grid": "3d7", "side": 75, "passes": 60},
        # many independent 2D systems, four right-hand sides each, one launch
        {"name": "batch_2d", "kind": "batch", "nsys": 608, "smin": 16, "smax": 96, "k": 0,
         "nrhs": 4, "mixed": True, "steps": 125},
        # same pattern, new coefficients: numeric refactorisation on the GPU
        {"name": "refactor_3d", "kind": "refactor", "grid": "3d7", "side": 101, "k": 1,
         "blocks": 64},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_blocks(rng, n):
    return rng.choice([b for b in (1, 2, 4, 8, 16, 32, 48, 64) if b == 1 or n // b >= 512])


def draw(rng):
    """One more case of the kinds and ranges above.  (``steps``: about what
    such a solve takes, for ``work``.)"""
    kind = rng.choice(["apply", "spmv", "projection", "gmres", "bicgstab", "cg", "batch", "refactor"])
    if kind == "projection":
        return {"kind": kind, "n": _log_int(rng, 2000, 2200000), "k": rng.randint(1, 31)}
    if kind == "batch":
        mixed = rng.random() < 0.7
        return {"kind": kind, "nsys": _log_int(rng, 8, 600 if mixed else 200), "smin": 16,
                "smax": rng.randint(20, 96), "k": rng.randint(0, 1), "nrhs": rng.randint(1, 4),
                "mixed": mixed, "steps": 60}
    grid = "3d7" if kind in ("cg", "bicgstab", "refactor") else rng.choice(["2d5", "3d7", "3d27i"])
    side = {"2d5": _log_int(rng, 32, 500), "3d7": _log_int(rng, 12, 128 if kind != "refactor" else 101),
            "3d27i": _log_int(rng, 12, 72)}[grid]
    n = side ** (2 if grid == "2d5" else 3)
    if kind == "spmv":
        return {"kind": kind, "grid": grid, "side": side, "f32": rng.random() < 0.5}
    if kind == "cg":
        return {"kind": kind, "grid": grid, "side": side, "passes": rng.randint(20, 60)}
    k = rng.randint(0, 2 if kind == "apply" else 1) if grid != "3d27i" else 0
    blocks = _draw_blocks(rng, n) if n <= 250000 else rng.choice([32, 48, 64])
    if kind == "apply":
        return {"kind": kind, "grid": grid, "side": side, "k": k, "blocks": blocks,
                "f32": rng.random() < 0.4}
    if kind == "bicgstab":
        return {"kind": kind, "grid": grid, "side": side, "k": k, "blocks": blocks,
                "passes": rng.randint(4, 16)}
    if kind == "refactor":
        return {"kind": kind, "grid": grid, "side": side, "k": k, "blocks": blocks}
    side = min(side, 160 if grid == "2d5" else 64)  # solved to convergence
    n = side ** (2 if grid == "2d5" else 3)
    return {"kind": kind, "grid": grid, "side": side, "k": k, "blocks": _draw_blocks(rng, n),
            "mixed": rng.random() < 0.5,
            "steps": 2 * side if grid == "2d5" else 30 + side if grid == "3d7" else 25}


# ------------------------------------------------------------------ inputs
_SIGMA = {"gmres": 0.5, "cg": 1.0, "bicgstab": 1.0}


def _matrix(case, seed):
    g, side = case["grid"], case["side"]
    sigma = _SIGMA.get(case["kind"], 2.0)
    if g == "2d5":
        return synth.diffusion2d_5pt_lognormal(side, sigma, seed)
    if g == "3d7":
        return synth.diffusion3d_7pt_lognormal(side, sigma, seed)
    return synth.stencil27_irregular(side, 2 * seed + 4, 2 * seed + 5)


def _batch(case, seed):
    """Systems of a batch: the sides follow from the case, the coefficients from the seed."""
    rng = np.random.default_rng(case["nsys"])
    sides = rng.integers(case["smin"], case["smax"] + 1, case["nsys"])
    seeds = np.random.default_rng(seed).integers(0, 2 ** 31 - 1, case["nsys"])
    return [synth.diffusion2d_5pt_lognormal(int(n), 0.5, int(c)) for n, c in zip(sides, seeds)]


def _uniform(shape, seed, dtype=torch.float64):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1000003 * int(seed) + 17)
    return torch.rand(shape, generator=gen, device="cuda", dtype=dtype) * 2 - 1


def _matvec(A, x):
    """A x in 64 bits, plain numpy (a row's terms side by side, one sum per
    row); x: a device tensor, one column or several."""
    xh = x.double().cpu().numpy()
    v = np.asarray(A.val)
    t = (v if xh.ndim == 1 else v[:, None]) * xh[np.asarray(A.col)]
    return torch.as_tensor(np.add.reduceat(t, np.asarray(A.row_ptr[:-1], np.int64), axis=0))


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": dict(case)}
    if kind == "projection":
        s["V"] = _uniform((case["k"], case["n"]), seed)
        s["w"] = _uniform((case["n"],), seed + 1)
        s["h"] = torch.empty(case["k"], device="cuda", dtype=torch.float64)
        return s
    if kind == "batch":
        mats = _batch(case, seed)
        s["B"] = H.hec_build_batched(mats)
        H.ilu_k_setup_batched(s["B"], case["k"])
        xt = _uniform((sum(A.n for A in mats), case["nrhs"]), seed)  # the solutions
        parts = xt.split([A.n for A in mats])
        s["b"] = torch.cat([_matvec(A, x) for A, x in zip(mats, parts)]).cuda()
        s["x"] = torch.zeros_like(s["b"])
        return s
    A = _matrix(case, seed)
    f32 = bool(case.get("f32"))
    dt = torch.float32 if f32 else torch.float64
    s["A"] = H.hec_build(A.row_ptr, A.col, A.val)
    if kind == "cg":
        s["M"] = H.jacobi_setup(s["A"], 1.0)
    elif kind != "spmv":
        s["M"] = H.ilu_k_setup(s["A"], case["k"], case["blocks"], 1 if case["blocks"] > 1 else 0)
        H.level_schedule(s["M"])
    x = _uniform((A.n,), seed, dt)
    if kind in ("apply", "spmv"):
        s["x"] = x
        s["y"] = torch.empty_like(x)
        s["w"] = _uniform((A.n,), seed + 1, dt)
        s["dots"] = torch.empty(2, device="cuda", dtype=torch.float64)
    elif kind == "gmres":
        s["b"] = _matvec(A, x).cuda()  # x is the solution
        s["x"] = torch.empty_like(x)
    elif kind in ("cg", "bicgstab"):
        s["b"] = x
        s["x"] = torch.empty_like(x)
    else:  # refactor: the coefficients come as a device array
        s["val"] = torch.as_tensor(A.val).cuda()
        s["r"] = x
        s["y"] = torch.empty_like(x)
        s["z"] = torch.empty_like(x)
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "projection":
        H.hec_multidot(case["n"], case["k"], s["V"], case["n"], s["w"], s["h"])
        return s["h"]
    if kind == "apply":
        f = H.hec_precond_apply_f32 if case["f32"] else H.hec_precond_apply
        f(s["M"], s["x"], s["y"])
        return s["y"]
    if kind == "spmv":
        if case["f32"]:
            H.hec_spmv_f32(s["A"], 1.0, s["x"], 0.0, None, s["y"])
            return s["y"]
        H.hec_spmv(s["A"], 1.0, s["x"], 0.0, None, s["y"], w=s["w"], dots=s["dots"])
        return s["y"], s["dots"]
    if kind == "gmres":
        H.krylov_solve(s["A"], s["M"], s["b"], s["x"], tol=1e-13, maxit=2000, restart=30,
                       method=H.GMRES, flags=H.X0_ZERO | (H.MIXED_FP32 if case["mixed"] else 0))
        return s["x"]
    if kind in ("cg", "bicgstab"):
        H.krylov_solve(s["A"], s["M"], s["b"], s["x"], tol=1e-14, maxit=case["passes"],
                       method=H.CG if kind == "cg" else H.BICGSTAB, flags=H.X0_ZERO)
        return s["x"]
    if kind == "batch":
        H.krylov_solve_batched(s["B"], s["b"], s["x"], nrhs=case["nrhs"], tol=1e-13, maxit=2000,
                               restart=30, flags=H.X0_ZERO | (H.MIXED_FP32 if case["mixed"] else 0))
        return s["x"]
    # the new values, then what the next time step needs of them at once
    H.hec_refactor(s["A"], s["M"], s["val"])
    H.hec_spmv(s["A"], 1.0, s["r"], 0.0, None, s["y"])
    H.hec_precond_apply(s["M"], s["r"], s["z"])
    return s["y"], s["z"]


# ------------------------------------------------------------------ work
def _sizes(case):
    """n, matrix entries, factor rows and factor entries (overlap and fill included)."""
    side, g = case["side"], case["grid"]
    n = side ** (2 if g == "2d5" else 3)
    nnz = {"2d5": 5 * n - 4 * side, "3d7": 7 * n - 6 * side * side,
           "3d27i": (3 * side - 2) ** 3 + round(0.02 * n) * 75}[g]
    k, blocks = case.get("k", 0), case.get("blocks", 1)
    # one layer of overlap on each side of a block's rows, at most the matrix;
    # the rows of one side only are needed in each of the two solves
    layer = 0 if blocks == 1 else (side if g == "2d5" else side * side)
    rows = min(n * blocks, n + blocks * layer)
    fill = {"2d5": (5, 7, 9), "3d7": (7, 13, 23), "3d27i": (27, 27, 27)}[g][k]
    return n, nnz, rows, rows * fill


def work(case):
    kind = case["kind"]
    if kind == "projection":
        n, k = case["n"], case["k"]
        return {"bytes": 8 * (k + 1) * n, "flops": 2 * k * n}
    if kind == "batch":
        lo, hi = case["smin"], case["smax"]
        n = case["nsys"] * (hi ** 3 - lo ** 3) / (3.0 * (hi - lo)) if hi > lo else case["nsys"] * lo * lo
        q, vb = case["nrhs"], 4 if case["mixed"] else 8
        # per step: matrix and factor entries once, their vectors, the basis
        # read for both projections (15 columns in the mean)
        step = n * ((5 + 5 + 2 * case["k"]) * (vb + 4) + q * vb * (6 + 2 * 15))
        flop = n * q * (2 * (10 + 2 * case["k"]) + 4 * 2 * 15)
        return {"bytes": int(case["steps"] * step), "flops": int(case["steps"] * flop)}
    n, nnz, rows, fnnz = _sizes(case)
    vb = 4 if case.get("f32") or case.get("mixed") else 8
    spmv = nnz * (vb + 4) + n * 2 * vb
    apply_ = fnnz * (vb + 4) + rows * (4 + vb) + n * 2 * vb
    if kind == "spmv":
        return {"bytes": spmv + (0 if case["f32"] else 8 * n), "flops": 2 * nnz + (0 if case["f32"] else 4 * n)}
    if kind == "apply":
        return {"bytes": apply_, "flops": 2 * fnnz}
    if kind == "gmres":
        step = spmv + apply_ + n * vb * (2 * 15 + 4)
        return {"bytes": case["steps"] * step, "flops": case["steps"] * (2 * nnz + 2 * fnnz + 4 * 2 * 15 * n)}
    if kind == "bicgstab":
        return {"bytes": case["passes"] * (2 * spmv + 2 * apply_ + 14 * 8 * n),
                "flops": case["passes"] * (4 * nnz + 4 * fnnz + 20 * n)}
    if kind == "cg":
        return {"bytes": case["passes"] * (spmv + 11 * 8 * n), "flops": case["passes"] * (2 * nnz + 12 * n)}
    # refactor: values in, slab and factor values out, then one SpMV and one apply
    return {"bytes": 8 * nnz * 2 + 12 * fnnz + 8 * fnnz + spmv + apply_,
            "flops": fnnz * (4 + 8 * case["k"]) + 2 * nnz + 2 * fnnz}


# ------------------------------------------------------------------ 64-bit values
def _ilu0_apply_2d5(A, side, r):
    """(LU)^-1 r for ILU(0) of a 5-point matrix, by anti-diagonals of the grid.
    The pattern has no triangles, so the elimination changes the diagonal only."""
    n = A.n
    rp, ci, va = np.asarray(A.row_ptr), np.asarray(A.col), np.asarray(A.val)
    rows = np.repeat(np.arange(n), np.diff(rp))
    off = {}
    for d in (-side, -1, 0, 1, side):
        v = np.zeros(n)
        m = ci - rows == d
        v[rows[m]] = va[m]
        off[d] = v
    i = np.arange(n)
    ix, iy = i % side, i // side
    fronts = [np.nonzero(ix + iy == f)[0] for f in range(2 * side - 1)]
    diag, y, z = off[0].copy(), r.copy(), np.zeros(n)
    for f in fronts:
        for d, ok in ((-side, iy[f] > 0), (-1, ix[f] > 0)):
            g = f[ok]
            lf = off[d][g] / diag[g + d]
            diag[g] -= lf * off[-d][g + d]
            y[g] -= lf * y[g + d]
    for f in reversed(fronts):
        s = y[f].copy()
        for d, ok in ((1, ix[f] < side - 1), (side, iy[f] < side - 1)):
            g = f[ok]
            s[ok] -= off[d][g] * z[g + d]
        z[f] = s / diag[f]
    return z


def exact(case, seed):
    kind = case["kind"]
    if kind == "projection":
        return _uniform((case["k"], case["n"]), seed) @ _uniform((case["n"],), seed + 1)
    if kind == "batch":  # the right-hand sides are A x for this x
        return _uniform((sum(A.n for A in _batch(case, seed)), case["nrhs"]), seed)
    if kind in ("cg", "bicgstab"):
        return None  # iterates of a budgeted solve
    if kind == "apply":
        if case["grid"] != "2d5" or case["k"] != 0 or case["blocks"] != 1:
            return None
        A = _matrix(case, seed)
        x = _uniform((A.n,), seed, torch.float32 if case["f32"] else torch.float64)
        return torch.as_tensor(_ilu0_apply_2d5(A, case["side"], x.double().cpu().numpy()))
    A = _matrix(case, seed)
    if kind == "gmres":
        return _uniform((A.n,), seed)
    x = _uniform((A.n,), seed, torch.float32 if case.get("f32") else torch.float64)
    y = _matvec(A, x).cuda()
    if kind == "refactor":
        return y, None
    if case["f32"]:
        return y
    w = _uniform((A.n,), seed + 1)
    return y, torch.stack([torch.dot(w, y), torch.dot(y, y)])
