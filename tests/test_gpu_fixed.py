"""The block fixed-point BiCGSTAB, CG and GMRES at the edges of its layouts and ranges, against the CPU oracle."""

import numpy as np
import pytest

import oracle
from paper_2308_08417_gb300 import workloads as W
from tests.parity import compare, host_rel_residual
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


def check(bbs, handle, pat, vals, b, fmt, x0=None, label="", **opts):
    A = W.make_batch(pat, vals, fmt)
    g = gpu_solve(bbs, handle, A, b, x0, **opts)
    r = oracle.solve_batch(A, b, x0, solver=opts.get("solver", "bicgstab"), restart=opts.get("gmres_restart", 10))
    D = W.to_dense(pat, vals).reshape(-1, pat.n, pat.n)
    fails = compare(*g[:4], r[0], r[1], r[3], rel_host=host_rel_residual(D, g[0], b), label=f"{label} {fmt} {opts}")
    assert not fails, "\n".join(fails)


@pytest.mark.parametrize("fmt", ["csr", "ell", "dense"])
@pytest.mark.parametrize("n", [66, 72])
def test_rows_longer_than_one_carry(bbs, handle, fmt, n):
    """Full rows: more than the 64 terms a product sums between carries, on one
    warp, on several and packed; n = 72 keeps dense digits by columns."""
    rng = np.random.default_rng(n)
    pat = W.random_pattern(n, n * n, rng)
    vals = W.general_values(pat, 5, rng, 0.05, 0.5)
    b = rng.uniform(-1, 1, (5, n))
    for tps in (16, 32, 64, 96):
        check(bbs, handle, pat, vals, b, fmt, threads_per_system=tps)


@pytest.mark.parametrize("fmt,tps", [("csr", 0), ("ell", 8), ("dense", 4), ("csr", 32), ("dense", 32)])
def test_fewer_rows_than_lanes_and_blocks_of_several_warps(bbs, handle, fmt, tps):
    """3 rows on 4 to 32 lanes, and batches that fill blocks of four warps with
    a ragged end (groups, and whole warps, without a system)."""
    rng = np.random.default_rng(7)
    for n, B in ((3, 21), (20, 6001)):
        if tps and -(-n // tps) > 10:
            continue
        pat = W.stencil_pattern("1d3", n)
        check(bbs, handle, pat, W.stencil_values(pat, B, rng, 0.05, 0.5), rng.uniform(-1, 1, (B, n)), fmt,
              threads_per_system=tps)


@pytest.mark.parametrize("tps", [0, 4, 32, 64])
@pytest.mark.parametrize("guess", [False, True])
def test_systems_that_do_not_fit_beside_ones_that_do(bbs, handle, tps, guess):
    """In one warp: systems scaled to the ends of FP64's range, one whose scaled
    rows sum to more than the fixed-point matrix holds, one with a zero guess
    among guesses of every size; each as the oracle solves it."""
    n, B = 40, 16
    rng = np.random.default_rng(3)
    pat = W.stencil_pattern("1d3", n)
    vals = W.stencil_values(pat, B, rng, 0.05, 0.5)
    b = rng.uniform(-1, 1, (B, n))
    rows = np.repeat(np.arange(n), np.diff(pat.row_ptrs))
    vals[1] *= 2.0 ** 480          # the matrix beyond FP32's range
    b[2] *= 2.0 ** 450             # the right-hand side beyond 2^400
    b[5] *= 2.0 ** -450
    r = np.where(np.arange(n) % 2, 64.0, 1.0)
    vals[9] *= r[rows]             # neighbouring rows scaled 64 : 1
    b[9] *= r
    b[12] *= 2.0 ** 390            # inside the range, at both ends
    b[13] *= 2.0 ** -390
    x0 = None
    if guess:
        D = W.to_dense(pat, vals).reshape(-1, n, n)
        x0 = np.linalg.solve(D, b[..., None])[..., 0] * (1 + 1e-3 * rng.uniform(-1, 1, (B, n)))
        x0[4] = 0.0
        x0[6] *= 1e6               # far from the solution
    check(bbs, handle, pat, vals, b, "csr", x0, threads_per_system=tps)


@pytest.mark.parametrize("fmt,tps", [("csr", 0), ("ell", 8), ("dense", 16), ("csr", 32), ("dense", 64), ("ell", 96)])
def test_cg_edges(bbs, handle, fmt, tps):
    """CG: 3 rows on many lanes, full rows longer than one carry, blocks of four
    warps with a ragged end, guesses, and in one batch systems that do not fit
    (a symmetric scaling of 64 : 1 between neighbours, both ends of the range)
    beside ones that do."""
    rng = np.random.default_rng(5)
    for n, B in ((3, 9), (20, 6001), (72, 5)):
        if tps and tps < 32 and -(-n // tps) > 10:
            continue
        if n == 72:  # a symmetric full matrix
            pat = W.random_pattern(n, n * n, rng)
            low = np.tril(rng.uniform(-1.0, 0.0, (B, n, n)), -1)
            full = low + low.transpose(0, 2, 1)
            i = np.arange(n)
            full[:, i, i] = np.abs(full).sum(2) * (1 + rng.uniform(0.05, 0.5, (B, n)))
            vals = full.reshape(B, -1)
        else:
            pat = W.stencil_pattern("1d3", n)
            vals = W.stencil_values(pat, B, rng, 0.05, 0.5, symmetric=True)
        check(bbs, handle, pat, vals, rng.uniform(-1, 1, (B, n)), fmt, solver="cg", threads_per_system=tps)
    n, B = 40, 12
    if tps == 0 or -(-n // tps) <= 10:
        pat = W.stencil_pattern("1d3", n)
        vals = W.stencil_values(pat, B, rng, 0.3, 0.9, symmetric=True)
        b = rng.uniform(-1, 1, (B, n))
        rows = np.repeat(np.arange(n), np.diff(pat.row_ptrs))
        r = np.where(np.arange(n) % 2, 64.0, 1.0)
        vals[3] *= r[rows] * r[pat.col_idxs]
        b[3] *= r
        vals[5] *= 2.0 ** 480
        b[6] *= 2.0 ** -450
        vals[8] *= 2.0 ** 90
        D = W.to_dense(pat, vals).reshape(-1, n, n)
        x0 = np.linalg.solve(D, b[..., None])[..., 0] * (1 + 1e-3 * rng.uniform(-1, 1, (B, n)))
        x0[4] = 0.0
        check(bbs, handle, pat, vals, b, fmt, x0, solver="cg", threads_per_system=tps)


@pytest.mark.parametrize("fmt,tps", [("csr", 0), ("ell", 4), ("dense", 8), ("csr", 16)])
@pytest.mark.parametrize("restart", [1, 10, 32])
def test_gmres_edges(bbs, handle, fmt, tps, restart):
    """GMRES: fewer rows than lanes, a heavy column (products above the rows' own
    bound), guesses, and systems that do not fit beside ones that do."""
    rng = np.random.default_rng(restart)
    pat = W.stencil_pattern("1d3", 3)
    check(bbs, handle, pat, W.stencil_values(pat, 9, rng, 0.3, 0.5), rng.uniform(-1, 1, (9, 3)), fmt, solver="gmres",
          threads_per_system=tps, gmres_restart=restart)
    n, B = 30, 13
    pat = W.random_pattern(n, n * n, rng)
    vals = W.general_values(pat, B, rng, 0.3, 0.9).reshape(B, n, n)
    vals[2, :, 4] = np.where(np.arange(n) == 4, vals[2, :, 4], 20.0 * vals[2, 4, 4])  # 29 entries of 20 a_jj
    vals = vals.reshape(B, -1)
    b = rng.uniform(-1, 1, (B, n))
    vals[5] *= 2.0 ** 480
    b[6] *= 2.0 ** -450
    vals[8] *= 2.0 ** 90
    D = W.to_dense(pat, vals).reshape(-1, n, n)
    x0 = np.linalg.solve(D, b[..., None])[..., 0] * (1 + 1e-3 * rng.uniform(-1, 1, (B, n)))
    x0[3] = 0.0
    A = W.make_batch(pat, vals, fmt)
    g = gpu_solve(bbs, handle, A, b, x0, threads_per_system=tps, solver="gmres", gmres_restart=restart, max_iters=400)
    r = oracle.solve_batch(A, b, x0, solver="gmres", restart=restart, max_iters=400)
    fails = compare(*g[:4], r[0], r[1], r[3], rel_host=host_rel_residual(D, g[0], b), label=f"gmres {fmt} {tps}")
    assert not fails, "\n".join(fails)


@pytest.mark.parametrize("solver,stencil,kx,ky,threads", [("bicgstab", "2d9", 13, 13, 64), ("bicgstab", "2d5", 16, 16, 64),
                                                          ("bicgstab", "1d3", 200, 1, 32), ("cg", "1d3", 200, 1, 64),
                                                          ("cg", "2d5", 13, 13, 32), ("bicgstab", "2d9", 18, 18, 64)])
def test_warps_per_system_do_not_depend_on_the_batch(bbs, handle, solver, stencil, kx, ky, threads):
    """The rule that gives long or many rows a second warp, on both sides of
    its line, and a system's bits in a batch of one and of many."""
    rng = np.random.default_rng(kx)
    pat = W.stencil_pattern(stencil, kx, ky) if ky > 1 else W.stencil_pattern(stencil, kx)
    sym = solver == "cg"
    vals = W.stencil_values(pat, 700, rng, 0.05, 0.5, **({"symmetric": True} if sym else {}))
    b = rng.uniform(-1, 1, (700, pat.n))
    few = 9
    check(bbs, handle, pat, vals[:few], b[:few], "csr", solver=solver)
    got = []
    for k in (few, 700):
        A = W.make_batch(pat, vals[:k], "csr")
        info = handle.describe(bbs.DeviceBatch.from_batch(A, "cuda"), bbs.bbs_default_options(solver=solver))
        assert info["threads_per_system"] == threads
        got.append(gpu_solve(bbs, handle, A, b[:k], solver=solver))
    for x, y in zip(got[0][:4], got[1][:4]):
        assert np.array_equal(x, y[:few])
