"""The packed kernels without a preconditioner, at the edges of their groups."""

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


@pytest.mark.parametrize("fmt", ["csr", "ell", "dense"])
@pytest.mark.parametrize("solver", ["bicgstab", "cg", "gmres"])
@pytest.mark.parametrize("tps,n", [(4, 3), (4, 40), (8, 63), (16, 17), (16, 33)])
def test_packed_without_preconditioner(bbs, handle, fmt, solver, tps, n):
    """Fewer rows than lanes, the most rows per lane, and one row past a group's
    width, in a batch with a ragged last warp; counts within 2 plus the oracle's own
    range under perturbations at rounding level."""
    rng = np.random.default_rng(n)
    pat = W.stencil_pattern("1d3", n)
    vals = W.stencil_values(pat, 37, rng, 0.3, 0.5, symmetric=True)
    b = rng.uniform(-1, 1, (37, n))
    A = W.make_batch(pat, vals, fmt)
    kw = dict(solver=solver, precond="none", max_iters=1000)
    g = gpu_solve(bbs, handle, A, b, None, threads_per_system=tps, **kw)
    r = oracle.solve_batch(A, b, None, **kw)
    D = W.to_dense(pat, vals).reshape(-1, n, n)
    fails = compare(*g[:4], r[0], r[1], r[3], rel_host=host_rel_residual(D, g[0], b), label=f"{fmt} {solver} {tps} {n}",
                    iter_tol=2 + iteration_spread(oracle.solve_batch, A, b, None, **kw))
    assert not fails, "\n".join(fails)
