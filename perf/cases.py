"""Performance cases: what a user of the library has it do, over its range.

A program analyses a sparsity pattern once, keeps the symbolic handle, and then
factors matrices of that pattern and solves with the factors:

    factor  new values, the factor itself is the result (the caller copies it)
    step    new values and new right-hand sides: refactor + solve (one time step,
            one Newton or optimisation step)
    solve   more right-hand sides for a factor that is kept

The matrices are the stencils of `paper_2409_13090_gb300.inputs` in the
benchmark's launch configuration (nested dissection with leaves of 8, partition
refinement, supernode merging 12.5 %), with values drawn anew from the seed. The
3D diffusion operators carry a diagonal term of 1e-2 (an implicit time step's
mass term; the shift that the library's own tests use on them).
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_2409_13090_gb300 as sc
from paper_2409_13090_gb300 import inputs

SHIFT = 1e-2


def _case(name, do, matrix, grid, precision, nrhs, variant="rlb", ordering="grid_nd", method="ir"):
    nx, ny, nz = grid
    c = {"do": do, "matrix": matrix, "nx": nx, "ny": ny, "nz": nz, "precision": precision, "nrhs": nrhs,
         "variant": variant, "ordering": ordering, "method": method}
    return {"name": name, **c} if name else c


def listed():
    return [
        # the smallest call: a 2D Poisson problem of 4,096 unknowns, one right-hand side
        _case("step_lap2d_64_fp64", "step", "lap2d", (64, 64, 1), "fp64", 1),
        # an odd-sized 2D problem with the RL variant; the caller takes the factor
        _case("factor_lap2d_83x71_fp64_rl", "factor", "lap2d", (83, 71, 1), "fp64", 0, variant="rl"),
        # ordinary time step of a variable-coefficient 3D diffusion, FP64
        _case("step_diff7_48_fp64", "step", "diff7", (48, 48, 48), "fp64", 4),
        # the same with the low-precision factor and conjugate gradients on top
        _case("step_diff7_48_tf32x3_cg", "step", "diff7", (48, 48, 48), "tf32x3", 4, method="cg"),
        # no coordinates and odd sides: the general-graph ordering, irregular supernodes
        _case("step_diff7_graph_37x41x29_fp64", "step", "diff7", (37, 41, 29), "fp64", 3, ordering="graph_ml"),
        # the largest FP64 step: 27-point stencil, 512,000 unknowns, 16 right-hand sides
        _case("step_st27_80_fp64", "step", "st27", (80, 80, 80), "fp64", 16),
        # the same in TF32 with classical refinement
        _case("step_st27_80_tf32", "step", "st27", (80, 80, 80), "tf32", 16),
        # 256 independent 2D problems of uneven size in one batch, FP32 + refinement
        _case("step_batch256_fp32", "step", "batch", (256, 32, 256), "fp32", 1),
        # the headline matrix: anisotropic 128^3, 64 right-hand sides, TF32x3 + conjugate gradients
        _case("step_aniso_128_tf32x3_cg", "step", "aniso", (128, 128, 128), "tf32x3", 64, method="cg"),
        # one more right-hand side for a kept FP64 factor (latency of the sweeps)
        _case("solve_diff7_48_fp64_1", "solve", "diff7", (48, 48, 48), "fp64", 1),
        # a block of 64 right-hand sides for a kept FP64 factor
        _case("solve_aniso_72x61x56_fp64_64", "solve", "aniso", (72, 61, 56), "fp64", 64),
        # many right-hand sides, a ragged count, FP32 factor + refinement
        _case("solve_st27_31x29x33_fp32_130", "solve", "st27", (31, 29, 33), "fp32", 130),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    do = rng.choice(["step", "step", "step", "solve", "factor"])
    precision = rng.choice(["fp64", "fp64", "fp64", "fp32", "tf32", "tf32x3"])
    if do == "factor":
        precision = "fp64"
    matrix = rng.choice(["lap2d", "diff7", "diff7", "st27", "aniso", "batch"])
    nrhs = 0 if do == "factor" else _log_int(rng, 1, 130)
    ordering, variant = "grid_nd", "rlb"
    if matrix == "lap2d":
        grid = (_log_int(rng, 24, 400), _log_int(rng, 24, 400), 1)
        variant = rng.choice(["rlb", "rl"])
    elif matrix == "batch":
        lo = _log_int(rng, 16, 64)
        grid = (_log_int(rng, 8, 160), lo, _log_int(rng, lo + 8, 200))
        nrhs = min(nrhs, 4)
    else:
        # about cubic, each side its own; the largest FP64 one costs less than the listed 80^3
        top = {"diff7": 72, "aniso": 72, "st27": 56}[matrix]
        if precision != "fp64":
            top = {"diff7": 96, "aniso": 96, "st27": 72}[matrix]
        side = _log_int(rng, 12, top)
        grid = tuple(max(8, min(top, int(round(side * rng.uniform(0.8, 1.2))))) for _ in range(3))
        n = grid[0] * grid[1] * grid[2]
        nrhs = min(nrhs, max(1, 40_000_000 // n)) if do != "factor" else 0
        if n <= 30_000:
            ordering = rng.choice(["grid_nd", "graph_ml"])
            variant = rng.choice(["rlb", "rlb", "rl"])
    method = rng.choice(["ir", "cg"]) if precision != "fp64" else "ir"
    return _case(None, do, matrix, grid, precision, nrhs, variant, ordering, method)


class _Problem:
    """What does not change with the values: patterns, the symbolic handle, and where A's entries lie."""

    def __init__(self, matrix, nx, ny, nz, variant, ordering):
        self.matrix = matrix
        kw = dict(ordering=ordering, variant=variant, merge=0.125)
        if matrix == "batch":  # nx matrices with sides from ny to nz
            sides = np.random.default_rng(nx).integers(ny, nz + 1, size=nx)
            parts = [inputs.laplacian_2d(int(s), int(s)) for s in sides]
            self.syms = [sc.Symbolic(A, grid=A.grid, **kw) for A in parts]
            self.sym = sc.Symbolic.batch(self.syms)
            self.flops = sum(s.view()["flops"] for s in self.syms)
            self.nnz_l = sum(int(s.view()["nnzL"]) for s in self.syms)
        else:
            A = {"lap2d": lambda: inputs.laplacian_2d(nx, ny),
                 "diff7": lambda: inputs.diffusion_3d_7pt(nx, ny, nz, 1),
                 "st27": lambda: inputs.stencil_3d_27pt(nx, ny, nz, 1),
                 "aniso": lambda: inputs.anisotropic_3d_7pt(nx, ny, nz, 1)}[matrix]()
            parts = [A]
            self.sym = sc.Symbolic(A, grid=A.grid if ordering == "grid_nd" else None, **kw)
            v = self.sym.view()
            self.flops, self.nnz_l = v["flops"], int(v["nnzL"])
        self.sizes = [A.n for A in parts]
        self.n = sum(self.sizes)
        row0 = np.concatenate([[0], np.cumsum(self.sizes)])[:-1]
        self.rows = np.concatenate([A.rowind.astype(np.int64) + r for A, r in zip(parts, row0)])
        self.cols = np.concatenate([np.repeat(np.arange(A.n, dtype=np.int64) + r, np.diff(A.colptr))
                                    for A, r in zip(parts, row0)])
        self.off = np.nonzero(self.rows != self.cols)[0]
        self.diag = np.nonzero(self.rows == self.cols)[0]
        self.along_z = (self.rows - self.cols)[self.off] == nx * ny
        self.nnz = len(self.rows)

    def values(self, seed):
        """A's entries (lower triangle, as analysed) for this seed."""
        rng = np.random.default_rng([seed, 20240913])
        r, c = self.rows[self.off], self.cols[self.off]
        v = np.empty(self.nnz)
        if self.matrix in ("lap2d", "batch"):  # unit couplings, each matrix with a shift of its own
            v[self.off] = -1.0
            v[self.diag] = 4.0 + np.repeat(rng.uniform(1e-3, 1e-1, len(self.sizes)), self.sizes)
            return v
        m = len(self.off)
        if self.matrix == "diff7":
            w = np.exp(rng.uniform(math.log(1e-2), math.log(1e2), m))
        elif self.matrix == "st27":
            w = rng.uniform(0.5, 1.5, m)
        else:
            w = np.where(self.along_z, 100.0, 1.0) * np.exp(rng.uniform(math.log(0.1), math.log(10.0), m))
        s = np.bincount(r, w, self.n) + np.bincount(c, w, self.n)
        v[self.off] = -w
        v[self.diag] = 1.01 * s if self.matrix == "st27" else s + SHIFT
        return v


@functools.lru_cache(maxsize=2)
def _cached(*key):
    return _Problem(*key)


def _problem(case):
    """One analysis serves every matrix of its pattern, as in a user's program."""
    return _cached(case["matrix"], case["nx"], case["ny"], case["nz"], case["variant"], case["ordering"])


def _rhs(p, nrhs, seed, device):
    g = torch.Generator(device=device)
    g.manual_seed(int(seed) * 7919 + 13)
    return torch.rand((nrhs, p.n), generator=g, device=device, dtype=torch.float64) * 2.0 - 1.0


def prepare(case, seed):
    p = _problem(case)
    values = torch.from_numpy(p.values(seed)).cuda()
    # the program's handle: created with a first matrix of the pattern (for "solve", the one that is kept)
    state = {"do": case["do"], "problem": p, "values": values, "method": case["method"],
             "factor": p.sym.factor(values, precision=case["precision"])}
    if case["do"] != "factor":
        state["B"] = _rhs(p, case["nrhs"], seed, "cuda")
        state["X"] = torch.empty_like(state["B"])
    return state


def run(state):
    num = state["factor"]
    if state["do"] != "solve":
        num.refactor(state["values"])
    if state["do"] == "factor":
        return {"L": num.device_view()["lnz"].clone()}  # the view ends with the handle: the caller keeps a copy
    X, _ = num.solve(state["B"], state["X"], method=state["method"], max_iterations=400)
    return {"X": X}


def work(case):
    p = _problem(case)
    low = case["precision"] != "fp64"
    elt = 4 if low else 8
    flops, nbytes = 0.0, 0.0
    if case["do"] != "solve":
        flops += p.flops
        nbytes += 8 * p.nnz + elt * p.nnz_l
    if case["do"] != "factor":
        # a forward and a backward sweep; a low-precision factor needs at least one correction more
        pairs = 2 if low else 1
        flops += 4.0 * pairs * p.nnz_l * case["nrhs"]
        nbytes += 2 * pairs * elt * p.nnz_l + 16 * p.n * case["nrhs"]
    return {"bytes": nbytes, "flops": flops}


def _dense(p, values):
    M = torch.zeros((p.n, p.n), dtype=torch.float64, device="cuda")
    r, c = torch.from_numpy(p.rows).cuda(), torch.from_numpy(p.cols).cuda()
    v = torch.from_numpy(values).cuda()
    M[r, c] = v
    M[c, r] = v
    return M


def _conjugate_gradients(p, values, B):
    """A X = B by Jacobi-preconditioned conjugate gradients in FP64, restarted from the true residual."""
    r = np.concatenate([p.rows, p.cols[p.off]])
    c = np.concatenate([p.cols, p.rows[p.off]])
    v = np.concatenate([values, values[p.off]])
    A = torch.sparse_coo_tensor(np.stack([r, c]), v, (p.n, p.n), device="cuda").coalesce().to_sparse_csr()
    dinv = 1.0 / torch.from_numpy(values[p.diag]).cuda()[:, None]
    b = B.T.contiguous()
    x = torch.zeros_like(b)
    norm = b.norm(dim=0)
    for _ in range(4):
        res = b - A @ x
        z = dinv * res
        d = z.clone()
        rz = (res * z).sum(0)
        start = res.norm(dim=0)
        for it in range(20000):
            q = A @ d
            a = rz / torch.clamp((d * q).sum(0), min=1e-300)
            x += a * d
            res -= a * q
            z = dinv * res
            rz2 = (res * z).sum(0)
            d = z + (rz2 / torch.clamp(rz, min=1e-300)) * d
            rz = rz2
            if it % 32 == 31 and bool((res.norm(dim=0) <= 1e-13 * torch.minimum(start, norm)).all()):
                break
    return x.T.contiguous()


def exact(case, seed):
    p = _problem(case)
    if case["do"] == "factor":
        if p.n > 8000:
            return None
        # dense Cholesky of the permuted matrix, laid out as the panels of the factor storage
        v = p.sym.view()
        perm = torch.from_numpy(v["perm"].astype(np.int64)).cuda()
        L = torch.linalg.cholesky(_dense(p, p.values(seed))[perm][:, perm]).cpu().numpy()
        num = p.sym.factor(p.values(seed), precision="fp64")
        d = num.device_view()
        out = np.zeros(d["lnz"].numel())
        for J, (f, e) in enumerate(zip(v["sup_ptr"][:-1], v["sup_ptr"][1:])):
            rows = v["glbind"][v["gl_ptr"][J]:v["gl_ptr"][J + 1]]
            block = np.where(rows[:, None] >= np.arange(f, e)[None, :], L[np.ix_(rows, np.arange(f, e))], 0.0)
            at = d["panel_off"][J] + np.arange(len(rows))[:, None] * d["panel_ld"][J] + np.arange(e - f)[None, :]
            out[at] = block
        return {"L": torch.from_numpy(out)}
    if p.n * case["nrhs"] > 16_000_000:
        return None
    return {"X": _conjugate_gradients(p, p.values(seed), _rhs(p, case["nrhs"], seed, "cuda"))}
