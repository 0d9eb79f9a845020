"""A kernel's dynamic shared-memory limit belongs to the function: calls of other
sizes through the same instance must leave it at the largest that was asked for."""

import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2308_08417_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bbs():
    from paper_2308_08417_gb300 import _build, bbs as mod

    _build.build()
    return mod


def test_two_threads_with_different_sizes(bbs):
    """Two host threads solve with the same packed instance (9 rows a lane: n = 144
    and 130, 64 and 58 KB a block): no launch of the larger finds the limit of the
    smaller."""
    o = bbs.bbs_default_options(max_iters=1)
    rng = np.random.default_rng(1)
    sides = []
    for kx, ky in ((12, 12), (13, 10)):
        pat, n = W.stencil_pattern("2d5", kx, ky), kx * ky
        A = bbs.DeviceBatch.from_batch(W.make_batch(pat, W.stencil_values(pat, 1300, rng, 0.05, 0.5), "csr"), "cuda")
        b = torch.as_tensor(rng.uniform(-1, 1, (1300, n)), device="cuda")
        h = bbs.Handle(0)
        info = h.describe(A, o)
        assert info["rows"] == 9 and info["smem"] > 48 * 1024
        sides.append((h, A, b, torch.zeros_like(b), bbs.Log.empty(1300), h.workspace(A, o), torch.cuda.Stream()))
    torch.cuda.synchronize()
    failed = []

    def work(h, A, b, x, log, ws, st):
        try:
            for _ in range(3000):
                h.solve(A, b, x, o, log, ws, stream=st)
        except bbs.BBSError as e:
            failed.append(str(e))

    threads = [threading.Thread(target=work, args=s) for s in sides]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not failed, failed


def test_large_network_after_a_small_one(bbs):
    """Prediction of a network made before a smaller one."""
    h = bbs.Handle(0)
    n, B = 144, 300
    rng = np.random.default_rng(2)
    pat = W.stencil_pattern("2d5", 12, 12)
    A = bbs.DeviceBatch.from_batch(W.make_batch(pat, W.stencil_values(pat, B, rng, 0.05, 0.5), "csr"), "cuda")
    b, xp, xn = (torch.as_tensor(rng.uniform(-1, 1, (B, n)), device="cuda") for _ in range(3))
    large = bbs.MLP(h, n, hidden=256, max_batch=4096)
    large.observe(A, b, xp, xn)
    large.finalize_stats()
    x0 = torch.empty_like(b)
    first = large.predict(A, b, xp, x0).clone()
    bbs.MLP(h, 16, hidden=64, max_batch=4096)
    assert torch.equal(large.predict(A, b, xp, x0), first)
