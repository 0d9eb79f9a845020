"""The block fixed-point solvers where the arithmetic is strained: weak diagonal
dominance, tight tolerances, entries of many sizes in one system."""

import numpy as np
import pytest

import oracle
from paper_2308_08417_gb300 import workloads as W
from tests.parity import host_rel_residual
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


@pytest.mark.parametrize("name", ["poisson", "poisson on two warps", "3-point", "9-point", "cg 3-point", "cg poisson"])
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
        pat, vals = recipe("1d3", 64, 1, 6000, *((1e-4, 1e-3) if solver == "cg" else (1e-3, 1e-2)), rng,
                           symmetric=solver == "cg")
    b = rng.uniform(-1, 1, (len(vals), pat.n))
    A = W.make_batch(pat, vals, "csr")
    x, it, rel, st = gpu_solve(bbs, handle, A, b, None, solver=solver, max_iters=2000)[:4]
    ref = oracle.solve_batch(A, b, None, solver=solver, max_iters=2000)
    assert (st[ref[3] == 0] == 0).all(), np.bincount(st)
    D = W.to_dense(pat, vals[:300]).reshape(-1, pat.n, pat.n)
    assert (rel[st == 0] <= 1e-10).all() and (host_rel_residual(D, x[:300], b[:300]) <= 1e-10 * (1 + 1e-6)).all()
