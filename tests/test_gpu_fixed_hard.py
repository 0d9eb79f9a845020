"""The block fixed-point solvers where the arithmetic is strained: weak diagonal
dominance, tight tolerances, entries of many sizes in one system."""

import numpy as np
import pytest

import oracle
from paper_2308_08417_gb300 import workloads as W
from tests.parity import compare, host_rel_residual, iteration_spread
from tests.test_gpu_parity import gpu_solve

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bbs():
    from paper_2308_08417_gb300 import _build, bbs as mod

    _build.build()
    return mod


@pytest.fixture(scope="module")
def handle(bbs):
    return bbs.Handle(0)


def tridiagonal(n, batch, diagonal):
    """batch copies of tridiag(-1, diagonal, -1)."""
    pat = W.stencil_pattern("1d3", n)
    rows = np.repeat(np.arange(n), np.diff(pat.row_ptrs))
    return pat, np.tile(np.where(pat.col_idxs == rows, diagonal, -1.0), (batch, 1))


def recipe(stencil, kx, ky, batch, lo, hi, rng, symmetric=False):
    pat = W.stencil_pattern(stencil, kx, ky) if ky > 1 else W.stencil_pattern(stencil, kx)
    return pat, W.stencil_values(pat, batch, rng, lo, hi, **({"symmetric": True} if symmetric else {}))


@pytest.mark.parametrize("name", ["poisson", "poisson on two warps", "9-point", "cg 3-point", "cg poisson"])
def test_weakly_dominant_systems_do_not_stop_early(bbs, handle, name):
    """Krylov vectors that cancel by many orders between two steps: every system
    that the FP64 oracle solves converges, to the tolerance."""
    rng = np.random.default_rng(11)
    solver = "cg" if name.startswith("cg") else "bicgstab"
    if "poisson" in name:
        pat, vals = tridiagonal(256 if "two" in name else 128, 300, 2.0)
    elif name == "9-point":
        pat, vals = recipe("2d9", 32, 32, 300, 1e-3, 1e-2, rng)
    else:
        pat, vals = recipe("1d3", 64, 1, 6000, 1e-4, 1e-3, rng, symmetric=True)
    b = rng.uniform(-1, 1, (len(vals), pat.n))
    A = W.make_batch(pat, vals, "csr")
    x, it, rel, st = gpu_solve(bbs, handle, A, b, None, solver=solver, max_iters=2000)[:4]
    ref = oracle.solve_batch(A, b, None, solver=solver, max_iters=2000)
    assert (st[ref[3] == 0] == 0).all(), np.bincount(st)
    D = W.to_dense(pat, vals[:300]).reshape(-1, pat.n, pat.n)
    assert (rel[st == 0] <= 1e-10).all() and (host_rel_residual(D, x[:300], b[:300]) <= 1e-10 * (1 + 1e-6)).all()


@pytest.mark.parametrize("name", ["poisson", "3-point"])
def test_weakly_dominant_systems_take_no_more_iterations(bbs, handle, name):
    """BiCGSTAB's count on such a system moves by several iterations under rounding
    alone, its mean over a batch hardly (6 / sqrt(300) of 270): within 1 % of the
    FP64 oracle's mean."""
    rng = np.random.default_rng(12)
    pat, vals = tridiagonal(256, 300, 2.0) if name == "poisson" else recipe("1d3", 64, 1, 6000, 1e-3, 2e-3, rng)
    b = rng.uniform(-1, 1, (len(vals), pat.n))
    A = W.make_batch(pat, vals, "csr")
    it = gpu_solve(bbs, handle, A, b, None, max_iters=2000)[1]
    ref = oracle.solve_batch(A, b, None, max_iters=2000)[1]
    assert it.mean() <= 1.01 * ref.mean(), (it.mean(), ref.mean())


def graded(name, n, batch, rng):
    """Systems whose equations have scales far apart: (pattern, values, b)."""
    pat = W.stencil_pattern("1d3", n)
    rows = np.repeat(np.arange(n), np.diff(pat.row_ptrs))
    off = pat.col_idxs != rows
    vals = W.stencil_values(pat, batch, rng, 0.3, 0.5, symmetric=True)
    b = rng.uniform(0.5, 1.0, (batch, n))
    if name == "diagonal":  # no coupling, right-hand sides from 1 to 1e-30
        vals[:, off] = 0.0
        b *= 10.0 ** -np.linspace(0, 30, n)
    elif name == "weakly coupled":
        vals[:, off] *= 1e-6
        b *= 10.0 ** -np.linspace(0, 20, n)
    else:  # two parts, the second in units 2^-30 or 2^-70 of the first's
        half = n // 2
        vals[:, (rows == half) & (pat.col_idxs < half)] = 0.0
        vals[:, (rows == half - 1) & (pat.col_idxs >= half)] = 0.0
        s = np.where(np.arange(n) < half, 1.0, 2.0 ** -int(name.split("^-")[1]))
        if name.startswith("rows"):
            vals = vals * s[rows]
        b = b * s
    return pat, vals, b


@pytest.mark.parametrize("tps", [0, 64])
@pytest.mark.parametrize("solver", ["bicgstab", "cg", "gmres"])
@pytest.mark.parametrize("guess", [False, True])
@pytest.mark.parametrize("name", ["diagonal", "weakly coupled", "rows 2^-30", "rows 2^-70", "b 2^-30", "b 2^-70"])
def test_small_entries_survive(bbs, handle, name, guess, solver, tps):
    """Each entry of x, not only the largest, is the oracle's to 1e-8: FP64 keeps
    an exponent per entry."""
    rng = np.random.default_rng(13)
    n, B = 24, 9
    pat, vals, b = graded(name, n, B, rng)
    if solver == "cg" and name.startswith("rows"):  # symmetric: the columns too
        s = np.where(np.arange(n) < n // 2, 1.0, 2.0 ** -int(name.split("^-")[1]))
        vals = vals * s[pat.col_idxs]
    A = W.make_batch(pat, vals, "csr")
    x0 = None
    if guess:
        x0 = oracle.solve_batch(A, b, None, solver=solver)[0] * (1 + 1e-3 * rng.uniform(-1, 1, (B, n)))
    x, _, _, st = gpu_solve(bbs, handle, A, b, x0, solver=solver, threads_per_system=tps)[:4]
    xr, _, _, sr = oracle.solve_batch(A, b, x0, solver=solver)[:4]
    assert np.array_equal(st, sr) and (sr == 0).all()
    assert (np.abs(x - xr) <= 1e-8 * np.abs(xr)).all(), np.abs(x / xr - 1).max()


@pytest.mark.parametrize("solver,fmt,tol", [("bicgstab", "csr", 1e-14), ("bicgstab", "ell", 4e-15), ("cg", "csr", 4e-15),
                                            ("gmres", "csr", 4e-15), ("bicgstab", "csr", 1e-10)])
def test_status_and_log_are_those_of_the_returned_x(bbs, handle, solver, fmt, tol):
    """At tolerances where rounding x to FP64 weighs: a system is CONVERGED only with
    a logged residual within the tolerance, and the log is the returned x's (to
    1e-3, or to the 1e-15 that FP64's own residual is good to)."""
    rng = np.random.default_rng(14)
    pat, vals = recipe("2d5", 12, 12, 8000, 0.05, 0.5, rng, symmetric=solver == "cg")
    b = rng.uniform(-1, 1, (len(vals), pat.n))
    x, _, rel, st = gpu_solve(bbs, handle, W.make_batch(pat, vals, fmt), b, None, solver=solver, tol=tol)[:4]
    assert (rel[st == 0] <= tol).all(), (int((rel[st == 0] > tol).sum()), rel[st == 0].max())
    pick = np.argsort(rel)[:: len(rel) // 200]
    D = W.to_dense(pat, vals[pick]).reshape(-1, pat.n, pat.n)
    rh = host_rel_residual(D, x[pick], b[pick])
    assert (np.abs(rel[pick] - rh) <= 1e-3 * rh + 1e-15).all()


@pytest.mark.parametrize("fmt,tps", [("csr", 0), ("ell", 4), ("dense", 16), ("csr", 32), ("ell", 64)])
@pytest.mark.parametrize("bits", [6, 20, 30])
def test_cg_with_diagonals_far_apart(bbs, handle, fmt, tps, bits):
    """Symmetric systems whose diagonal entries lie 2^bits apart (inside the range of
    the weights, near its end and beyond it), as a 3-point batch has them at its
    corners: the oracle's x, iterations and status."""
    rng = np.random.default_rng(bits)
    n, B = 40, 33
    pat, vals = recipe("1d3", n, 1, B, 0.05, 0.5, rng, symmetric=True)
    rows = np.repeat(np.arange(n), np.diff(pat.row_ptrs))
    s = np.ones((B, n))
    s[np.arange(B), rng.integers(0, n, B)] = 2.0 ** (-bits / 2)  # one small row and column
    vals = vals * s[:, rows] * s[:, pat.col_idxs]
    b = rng.uniform(-1, 1, (B, n)) * s
    for x0 in (None, rng.uniform(-1, 1, (B, n))):
        A = W.make_batch(pat, vals, fmt)
        g = gpu_solve(bbs, handle, A, b, x0, solver="cg", threads_per_system=tps)
        r = oracle.solve_batch(A, b, x0, solver="cg")
        D = W.to_dense(pat, vals).reshape(-1, n, n)
        fails = compare(*g[:4], r[0], r[1], r[3], rel_host=host_rel_residual(D, g[0], b), label=f"{fmt} {tps}",
                        iter_tol=2 + iteration_spread(oracle.solve_batch, A, b, x0, solver="cg"))
        assert not fails, "\n".join(fails)


@pytest.mark.parametrize("solver", ["bicgstab", "cg", "gmres"])
@pytest.mark.parametrize("tps,tol", [(4, 1e-10), (4, 2e-15), (8, 2e-15), (16, 2e-15)])
def test_bits_do_not_depend_on_the_warps_other_systems(bbs, handle, solver, tps, tol):
    """Systems whose residuals fall by 1 to 40 bits a step, restart, break down or do not
    fit, in one batch: each keeps its bits wherever it stands in it."""
    rng = np.random.default_rng(19)
    n, B = 30, 4000
    pat, vals = recipe("1d3", n, 1, B, 0.01, 0.02, rng, symmetric=True)
    rows = np.repeat(np.arange(n), np.diff(pat.row_ptrs))
    diag = pat.col_idxs == rows
    vals[:, diag] *= 10.0 ** (6 * rng.uniform(0, 1, (B, 1)) ** 3)
    b = rng.uniform(-1, 1, (B, n))
    b[::7] *= 2.0 ** -(30 * rng.uniform(0, 1, (len(b[::7]), n)))
    x0 = np.where(rng.uniform(0, 1, (B, 1)) < 0.3, rng.uniform(-1, 1, (B, n)), 0.0)
    kw = dict(solver=solver, threads_per_system=tps, tol=tol, max_iters=200)
    want = gpu_solve(bbs, handle, W.make_batch(pat, vals, "ell"), b, x0, **kw)
    for _ in range(3):
        p = rng.permutation(B)
        got = gpu_solve(bbs, handle, W.make_batch(pat, vals[p], "ell"), b[p], x0[p], **kw)
        for w, g in zip(want[:4], got[:4]):
            assert np.array_equal(w[p], g, equal_nan=w.dtype.kind == "f")
