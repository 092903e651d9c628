"""FP64 products on the tensor cores as products of FP16 slices (needs a GB300).

The sizes are the edges of the path: inner dimensions around a 32-column stage
and around the 128 columns between two drains of the accumulators, row and
column counts around the 128 x 64 tile, chunk widths that start a product's
columns at 24 (16-byte aligned) or 33 (not: such products stay on the SIMT
tiles), rows of very different scale, and a row holding a NaN.

Tolerance: a factor entry is sqrt-sized against its row, |L_ij| <= sqrt(a_ii); the
oracle's own rounding of n sequential multiply-adds is below n u sqrt(a_ii), so the
two agree within 2 n u sqrt(a_ii) (n <= 700, u = 2^-53: 1.6e-13), here 1e-12.
"""
import numpy as np
import pytest

import oracle
import paper_2409_13090_gb300 as sc
from paper_2409_13090_gb300 import inputs
from tests.test_gpu_tc import _dense

pytestmark = pytest.mark.gpu
TOL = 1e-12


@pytest.fixture(scope="module", autouse=True)
def built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    sc.build()
    oracle.build()


def _row_scale(A):
    d = A.values[A.colptr[:-1]]  # natural ordering: the diagonal is first in its column
    return np.sqrt(d)[np.repeat(np.arange(A.n), A.n)]


def _factors(A, **kw):
    sym = sc.Symbolic(A, ordering="natural", **kw)
    assert sym.check_schedule()["ok"]
    num = sym.factor(A.values, precision="fp64")
    return sym, num, num.profile(A.values)["gemm_tc"]["launches"]


@pytest.mark.parametrize("chunk", [64, 24, 33])
@pytest.mark.parametrize("n", [97, 128, 129, 191, 193, 257, 320, 385, 700])
def test_dense_sizes_around_the_tiles(n, chunk):
    A = _dense(n, n)
    sym, num, launches = _factors(A, chunk=chunk)
    assert num.rc == 0 and (launches > 0 or n < 128)
    o = oracle.Oracle(A, None, pr=True)
    assert o.factor() == 0
    err = np.abs(num.export_L() - o.L_supernodal())
    assert (err <= TOL * _row_scale(A)).all(), err.max()


def test_rows_of_very_different_scale():
    """D A D with D = 2^-60 .. 2^60 in random order: the factor is D L, every row
    to the accuracy of its own scale (the scaling itself is exact)."""
    A = _dense(300, 5)
    d = 2.0 ** np.random.default_rng(3).integers(-60, 61, size=A.n)
    cols = np.repeat(np.arange(A.n), np.diff(A.colptr))
    A.values *= d[A.rowind] * d[cols]
    _, num, launches = _factors(A)
    assert num.rc == 0 and launches > 0
    o = oracle.Oracle(A, None, pr=True)
    assert o.factor() == 0
    err = np.abs(num.export_L() - o.L_supernodal())
    assert (err <= TOL * _row_scale(A)).all()


@pytest.mark.parametrize("scaled_rhs", [True, False])
@pytest.mark.parametrize("nrhs", [1, 9, 33])
def test_solve_with_rows_of_very_different_scale(nrhs, scaled_rhs):
    """(D A D) x = b: with b = D b0 the solution is D^{-1} (A^{-1} b0), every entry to the
    accuracy of its own scale (A is diagonally dominant; 2 n u rounded up to
    1e-12 of the largest entry of A^{-1} b0). With b = b0 the right-hand side D^{-1} b0
    has entries of very different size, and the comparison is by the largest."""
    A = _dense(300, 5)
    d = 2.0 ** np.random.default_rng(3).integers(-60, 61, size=A.n)
    b0 = inputs.rhs(A.n, nrhs, 4) / (1.0 if scaled_rhs else d[:, None])
    o = oracle.Oracle(A, None, pr=True)
    assert o.factor() == 0
    x0 = o.solve(b0)
    cols = np.repeat(np.arange(A.n), np.diff(A.colptr))
    A.values *= d[A.rowind] * d[cols]
    num = sc.Symbolic(A, ordering="natural").factor(A.values, precision="fp64")
    X, _ = num.solve(b0 * d[:, None])
    assert np.abs(X * d[:, None] - x0).max() <= 1e-12 * np.abs(x0).max()


def test_nan_reaches_the_pivot():
    """A NaN in A's first column at row 200 of 300: rows below row 200 and the
    pivot of column 201 (1-based) see it, the columns before do not."""
    A = _dense(300, 6)
    v = A.values.copy()
    v[A.colptr[0] + 200] = np.nan
    sym = sc.Symbolic(A, ordering="natural")
    num = sym.factor(v, precision="fp64")
    assert num.rc == 201
    good = sym.factor(A.values, precision="fp64")
    L, G = num.export_L().reshape(300, 300), good.export_L().reshape(300, 300)
    assert np.abs(L[:200, :200] - G[:200, :200]).max() <= TOL * np.abs(G).max()


@pytest.mark.parametrize("variant", ["rlb", "rl"])
def test_irregular_updates_between_supernodes(variant):
    """Products into ancestors (atomic adds, or update matrices stored and then
    assembled) of a 3D 27-point matrix, merged and not."""
    A = inputs.stencil_3d_27pt(13, 11, 12, seed=9)
    for merge in (0.0, 0.3):
        sym = sc.Symbolic(A, ordering="grid_nd", grid=A.grid, variant=variant, merge=merge)
        assert sym.check_schedule()["ok"]
        num = sym.factor(A.values, precision="fp64")
        p = num.profile(A.values)
        assert num.rc == 0 and p["gemm_tc"]["launches"] > 0
        o = oracle.Oracle(A, oracle.nd_grid(*A.grid, 8), pr=True, merge=merge)
        assert o.factor() == 0
        Lo = o.L_supernodal()
        num.refactor(A.values)
        assert np.abs(num.export_L() - Lo).max() <= TOL * np.abs(Lo).max()


@pytest.mark.parametrize("blocks", [600, 3000])
def test_pivot_roots_over_the_exponent_range(blocks):
    """2 x 2 blocks [[d, a], [a, e]] with d from 2^-1000 to 2^1000 (both sides of where
    the POTRFs' approximations give way to the library's functions), by the CTA-wide
    POTRF (600 chunks on the level) and by warps (3000). With u = 2^-53: 1 / sqrt(d)
    has one rounding in e's product d y (half of it counts) and one at the end, 1.5 u
    and less than 2^-58 of the series; sqrt(d) = d rk one more: below 3 u (the
    library's 1 / sqrt(d), 2 u: 3 u; 3.1 u with the reference's long double). L_10 is
    a rk, 3 u, or (a / d) sqrt(d): 2 u, 3 u and one more product, 6 u; 6.2 u with the
    products of these errors."""
    rng = np.random.default_rng(blocks)
    d = np.ldexp(rng.uniform(1.0, 2.0, blocks), rng.integers(-1000, 1001, blocks))
    d[:6] = np.ldexp(1.0, [-1000, -991, -990, 991, 993, 1000])
    a = d * rng.uniform(-0.5, 0.5, blocks)  # a^2 / d < d
    n = 2 * blocks
    values = np.stack([d, a, d], 1).ravel()
    even = np.arange(0, n, 2)
    colptr = np.append(np.stack([even // 2 * 3, even // 2 * 3 + 2], 1).ravel(), 3 * blocks)
    A = inputs.SparseSym(n, colptr.astype(np.int64), np.stack([even, even + 1, even + 1], 1).ravel().astype(np.int32), values)
    num = sc.Symbolic(A, ordering="natural").factor(A.values, precision="fp64")
    assert num.rc == 0
    L = num.export_L()
    root = np.sqrt(d.astype(np.longdouble))
    u = 2.0 ** -53
    L = L.reshape(blocks, 2, 2)
    assert (np.abs(L[:, 0, 0] - root) <= 3.1 * u * root).all()
    ref = a / root
    assert (np.abs(L[:, 1, 0] - ref) <= 6.2 * u * np.abs(ref)).all()


@pytest.mark.parametrize("chunk", [17, 31, 32, 33, 48, 49, 63, 64])
def test_solve_by_inverses_of_every_width(chunk):
    """Diagonal blocks of one to four 16-column panels, whole and ragged, and a last chunk
    of another width. Diagonally dominant, so 2 n u of the largest entry rounded up to 1e-12."""
    A = _dense(170, chunk)
    B = inputs.rhs(A.n, 9, chunk)
    o = oracle.Oracle(A, None, pr=True)
    assert o.factor() == 0
    x0 = o.solve(B)
    X, _ = sc.Symbolic(A, ordering="natural", chunk=chunk).factor(A.values, precision="fp64").solve(B)
    assert np.abs(X - x0).max() <= 1e-12 * np.abs(x0).max()


@pytest.mark.parametrize("lookahead", [1, -1])
@pytest.mark.parametrize("matrix", ["st27", "lap2d"])
def test_profile_of_a_fused_handle(matrix, lookahead):
    """A handle with one launch per level holds no digits: its profile runs the FP64-pipe kernels
    of its own plan, class by class, and leaves the factor. Bound: the module's."""
    A = inputs.stencil_3d_27pt(13, 11, 12, seed=9) if matrix == "st27" else inputs.laplacian_2d(37, 29, 0.05)
    sym = sc.Symbolic(A, ordering="grid_nd", grid=A.grid, merge=0.3, tune=dict(fused=1, lookahead=lookahead))
    num = sym.factor(A.values, precision="fp64")
    p = num.profile(A.values)
    assert p["potrf"]["launches"] > 0 and p["trsm"]["launches"] > 0 and p["rlb_loop"]["launches"] > 0
    assert p["gemm_tc"]["launches"] == 0
    o = oracle.Oracle(A, oracle.nd_grid(*A.grid, 8), pr=True, merge=0.3)
    assert o.factor() == 0
    Lo = o.L_supernodal()
    assert np.abs(num.export_L() - Lo).max() <= TOL * np.abs(Lo).max()


def _dense_sym(M):
    n = len(M)
    cols = np.concatenate([[0], np.cumsum(np.arange(n, 0, -1))]).astype(np.int64)
    rows = np.concatenate([np.arange(j, n) for j in range(n)]).astype(np.int32)
    return inputs.SparseSym(n, cols, rows, np.concatenate([M[j:, j] for j in range(n)]))


def _kernel_matrix(n, length, nugget):
    """Gaussian kernel on n equally spaced points of [0, 1]: its leading blocks are
    as ill-conditioned as the nugget allows (2-norm condition about n / nugget)."""
    t = np.linspace(0.0, 1.0, n)
    return np.exp(-0.5 * ((t[:, None] - t) / length) ** 2) + nugget * np.eye(n)


@pytest.mark.parametrize("n,chunk", [(192, 64), (150, 64), (192, 24), (131, 33)])
@pytest.mark.parametrize("nugget", [1e-2, 1e-5, 1e-8, 1e-11, 1e-13])
@pytest.mark.parametrize("length", [0.02, 0.1])
def test_factor_of_ill_conditioned_blocks(length, nugget, n, chunk):
    """|A - L L^T| <= (n + 1) u sqrt(a_ii a_jj): the bound of Cholesky in FP64 (Higham, "Accuracy and
    Stability of Numerical Algorithms", 10.3, with |L| |L|^T <= sqrt(a_ii a_jj)), whatever
    the condition; and no pivot <= 0 where the oracle finds none."""
    M = _kernel_matrix(n, length, nugget)
    A = _dense_sym(M)
    o = oracle.Oracle(A, None, pr=True)
    assert o.factor() == 0
    sym = sc.Symbolic(A, ordering="natural", chunk=chunk)
    num = sym.factor(A.values, precision="fp64")
    assert num.rc == 0
    v = sym.view()
    perm = np.asarray(v["perm"], dtype=np.int64)
    assert v["nsuper"] == 1
    L = np.tril(num.export_L().reshape(n, n)).astype(np.longdouble)
    P = M[np.ix_(perm, perm)]
    d = np.sqrt(np.diag(P))
    res = np.abs(P.astype(np.longdouble) - L @ L.T) / np.outer(d, d)
    assert res.max() <= (n + 1) * 2.0 ** -53


@pytest.mark.parametrize("nrhs", [1, 9, 20, 33, 70])
@pytest.mark.parametrize("what,n,chunk", [("1e-8", 192, 64), ("1e-11", 150, 33), ("1e-13", 192, 24), ("1e-5", 131, 64),
                                          ("fourth difference", 1024, 64)])
def test_solve_with_ill_conditioned_blocks(what, n, chunk, nrhs):
    """Gaussian kernels with a nugget, and the 1D fourth difference as one supernode: the plain FP64
    solve (no refinement) is backward stable, eta <= 1e-14 (the default ir_tol; n u is 1.5e-14 to
    1.1e-13), for right-hand sides of smooth, random and random A x."""
    if what == "fourth difference":
        M = sum(c * np.eye(n, k=k) for k, c in ((-2, 1.0), (-1, -4.0), (0, 6.0), (1, -4.0), (2, 1.0)))
    else:
        M = _kernel_matrix(n, 0.05, float(what))
    A = _dense_sym(M)
    rng = np.random.default_rng(nrhs)
    B = rng.uniform(-1.0, 1.0, (n, nrhs))
    B[:, ::3] = M @ B[:, ::3]
    B[:, 1::3] = np.cos(np.arange(n) / n * np.arange(1, nrhs + 1)[1::3, None]).T
    num = sc.Symbolic(A, ordering="natural", chunk=chunk).factor(A.values, precision="fp64")
    assert num.rc == 0
    X, info = num.solve(B)
    eta = oracle.backward_error(A, B, X)
    assert eta.max() <= 1e-14, eta.max()
    assert info["converged"] and info["iterations"] == 0


@pytest.mark.parametrize("what", ["dense 700", "dense 700 chunk 24", "deterministic st27", "deterministic lap2d"])
def test_products_without_the_slice_pool(what):
    """A handle without memory for the slices forms the same products from the panels: the same
    bits where the additions have one order (one supernode; deterministic plans)."""
    if what.startswith("dense"):
        A = _dense(700, 3)
        sym = sc.Symbolic(A, ordering="natural", chunk=24 if "24" in what else 64)
    else:
        A = inputs.stencil_3d_27pt(13, 11, 12, seed=9) if "st27" in what else inputs.laplacian_2d(83, 71, 0.05)
        sym = sc.Symbolic(A, ordering="grid_nd", grid=A.grid, merge=0.3, variant="rl", deterministic=True)
    num = sym.factor(A.values, precision="fp64")
    p = num.profile(A.values)
    assert num.rc == 0 and (p["gemm_tc"]["launches"] > 0 or what.endswith("lap2d"))
    L = num.export_L()
    try:
        num.drop_slices()
    except sc.SCError:
        assert p["gemm_tc"]["launches"] == 0  # no product large enough
        return
    num.refactor(A.values)
    assert np.array_equal(num.export_L().view(np.uint64), L.view(np.uint64))
    with pytest.raises(sc.SCError):
        num.drop_slices()
    num.refactor(A.values)
    assert np.array_equal(num.export_L().view(np.uint64), L.view(np.uint64))


@pytest.mark.parametrize("variant", ["rlb", "rl"])
def test_irregular_updates_without_the_slice_pool(variant):
    """As test_irregular_updates_between_supernodes, by the products from the panels."""
    A = inputs.stencil_3d_27pt(13, 11, 12, seed=9)
    sym = sc.Symbolic(A, ordering="grid_nd", grid=A.grid, variant=variant, merge=0.3)
    num = sym.factor(A.values, precision="fp64")
    num.drop_slices()
    num.refactor(A.values)
    o = oracle.Oracle(A, oracle.nd_grid(*A.grid, 8), pr=True, merge=0.3)
    assert o.factor() == 0
    Lo = o.L_supernodal()
    assert np.abs(num.export_L() - Lo).max() <= TOL * np.abs(Lo).max()


@pytest.mark.parametrize("nrhs", [1, 5, 20, 33, 70])
@pytest.mark.parametrize("n", [64, 200])
def test_decaying_solutions_of_a_fused_handle(n, nrhs):
    """tune.fused = 1 is FP64 operations throughout, also in the solve: a chain of 4 on the
    diagonal and -1 beside it, as one supernode, with a unit right-hand side. The solution decays by
    3.7 a step, and nothing cancels in it: every entry has a relative error below 3 u per
    step and sweep (one division, one product, one rounding) on top of the factor's 3 u
    per pivot, below 9 n u in all; 10 n u."""
    A = _dense_sym(4.0 * np.eye(n) - np.eye(n, k=1) - np.eye(n, k=-1))
    B = np.zeros((n, nrhs))
    B[np.arange(nrhs) * 3 % n, np.arange(nrhs)] = 1.0
    num = sc.Symbolic(A, ordering="natural", pr=False, tune=dict(fused=1)).factor(A.values, precision="fp64")
    assert num.rc == 0
    X, _ = num.solve(B)
    # the same elimination in long double
    one = np.longdouble(1)
    d, x = np.empty(n, np.longdouble), B.astype(np.longdouble)
    d[0] = 4
    for i in range(1, n):
        d[i] = 4 - one / d[i - 1]
        x[i] += x[i - 1] / d[i - 1]
    x[-1] /= d[-1]
    for i in range(n - 2, -1, -1):
        x[i] = (x[i] + x[i + 1]) / d[i]
    assert (np.abs(X - x) <= 10 * n * 2.0 ** -53 * np.abs(x)).all()


@pytest.mark.parametrize("nrhs", [1, 2, 4, 7, 16, 31, 64, 130])
@pytest.mark.parametrize("matrix", ["st27", "dense"])
def test_solve_of_a_fused_handle(matrix, nrhs):
    """Substitution with every register layout of the right-hand sides, against the oracle (2 n u of
    the largest entry rounded up to 1e-12: both matrices are diagonally dominant)."""
    A = inputs.stencil_3d_27pt(13, 11, 12, seed=9) if matrix == "st27" else _dense(170, 7)
    kw = dict(ordering="grid_nd", grid=A.grid, merge=0.3) if matrix == "st27" else dict(ordering="natural", chunk=33)
    o = oracle.Oracle(A, oracle.nd_grid(*A.grid, 8) if matrix == "st27" else None, pr=True)
    assert o.factor() == 0
    B = inputs.rhs(A.n, nrhs, nrhs)
    x0 = o.solve(B)
    X, _ = sc.Symbolic(A, tune=dict(fused=1), **kw).factor(A.values, precision="fp64").solve(B)
    assert np.abs(X - x0).max() <= 1e-12 * np.abs(x0).max()


@pytest.mark.parametrize("blocks", [600, 3000])
def test_second_pivots_over_the_exponent_range(blocks):
    """The 2 x 2 blocks of test_pivot_roots_over_the_exponent_range, [[d, a], [a, d]] with |a| <=
    d / 2: L_11 = sqrt(d - a^2 / d) passes through the updated column. By the CTA-wide POTRF
    a / d has 2 u and its product with a one FMA: (2 u a^2 / d) / (d - a^2 / d) + u <= 5/3 u;
    by warps L_10 has 3 u, L_10^2 6 u: at most 3 u. Half of it in the root, whose own
    error is 3 u: 4.5 u, 4.6 u with the products of these errors."""
    rng = np.random.default_rng(blocks)
    d = np.ldexp(rng.uniform(1.0, 2.0, blocks), rng.integers(-1000, 1001, blocks))
    d[:6] = np.ldexp(1.0, [-1000, -991, -990, 991, 993, 1000])
    a = d * rng.uniform(-0.5, 0.5, blocks)
    n = 2 * blocks
    even = np.arange(0, n, 2)
    colptr = np.append(np.stack([even // 2 * 3, even // 2 * 3 + 2], 1).ravel(), 3 * blocks)
    A = inputs.SparseSym(n, colptr.astype(np.int64), np.stack([even, even + 1, even + 1], 1).ravel().astype(np.int32),
                         np.stack([d, a, d], 1).ravel())
    num = sc.Symbolic(A, ordering="natural").factor(A.values, precision="fp64")
    assert num.rc == 0
    L = num.export_L().reshape(blocks, 2, 2)[:, 1, 1]
    dl, al = d.astype(np.longdouble), a.astype(np.longdouble)
    ref = np.sqrt(dl - al / dl * al)
    assert (np.abs(L - ref) <= 4.6 * 2.0 ** -53 * ref).all()


@pytest.mark.parametrize("wa,wc,wb", [(5, 3, 40), (1, 2, 17), (7, 6, 90), (4, 8, 31)])
def test_small_chunks_with_rows_below(wa, wc, wb):
    """600 problems of two leaves (wa and wc columns) under one root of wb: 1200 small chunks on a
    level, taken by a warp each, with the rows below them in whole and ragged runs of 32, and rows
    of very different scale. L against the oracle's, row by row."""
    blocks, nb = 600, wa + wc + wb
    rng = np.random.default_rng(wb)
    M = np.zeros((nb, nb), dtype=bool)
    for s in (slice(0, wa), slice(wa, wa + wc)):
        M[s, s] = M[wa + wc:, s] = True
    M[wa + wc:, wa + wc:] = True
    r, c = np.nonzero(np.tril(M).T)[::-1]  # by columns
    per = np.bincount(c, minlength=nb)
    rows = (r[None, :] + nb * np.arange(blocks)[:, None]).ravel()
    colptr = np.concatenate([[0], np.cumsum(np.tile(per, blocks))])
    cols = (c[None, :] + nb * np.arange(blocks)[:, None]).ravel()
    v = rng.uniform(-1.0, 1.0, len(rows))
    n = blocks * nb
    v[rows == cols] = 2.0 * nb
    d = 2.0 ** rng.integers(-40, 41, size=n)
    A = inputs.SparseSym(n, colptr.astype(np.int64), rows.astype(np.int32), v * d[rows] * d[cols])
    sym = sc.Symbolic(A, ordering="natural")
    v = sym.view()
    widths = np.diff(v["sup_ptr"])
    assert v["nsuper"] == 3 * blocks and sorted(set(widths)) == sorted({wa, wc, wb})
    num = sym.factor(A.values, precision="fp64")
    assert num.rc == 0
    o = oracle.Oracle(A, None, pr=True)
    assert o.factor() == 0
    diag = np.empty(n)
    diag[A.rowind[A.colptr[:-1]]] = A.values[A.colptr[:-1]]
    scale = np.concatenate([np.repeat(np.sqrt(diag[v["perm"]][v["glbind"][v["gl_ptr"][J]:v["gl_ptr"][J + 1]]]),
                                      widths[J]) for J in range(v["nsuper"])])
    assert (np.abs(num.export_L() - o.L_supernodal()) <= TOL * scale).all()


def test_without_memory_for_the_inverses():
    """With less device memory than FP64 by digits holds beside the factor (all but that much is
    taken first), an RLB handle runs by FP64 operations."""
    import torch
    A = inputs.laplacian_2d(1000, 1000, 0.05)
    kw = dict(ordering="grid_nd", grid=A.grid, merge=0.125)
    sym = sc.Symbolic(A, **kw)
    B = inputs.rhs(A.n, 2, 1)
    num = sym.factor(A.values, precision="fp64")
    full = num.info.device_bytes
    X0, _ = num.solve(B)
    num.free()
    small = sc.Symbolic(A, tune=dict(fused=1), **kw).factor(A.values, precision="fp64").info.device_bytes
    assert full - small > 160 << 20
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    taken = torch.empty(free - small - (64 << 20), dtype=torch.uint8, device="cuda")
    try:
        num = sym.factor(A.values, precision="fp64")
        assert num.rc == 0 and num.info.device_bytes < full - (128 << 20)
    finally:
        del taken
        torch.cuda.empty_cache()
    X, _ = num.solve(B)
    assert np.abs(X - X0).max() <= TOL * np.abs(X0).max()
    assert num.profile(A.values)["gemm_tc"]["launches"] == 0
