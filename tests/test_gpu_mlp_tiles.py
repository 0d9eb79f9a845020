"""The training step's kernels at the edges of their tiles (128 rows, up to 64
columns, 64 of K; weight gradients split over K or whole): the tcgen05 path
against the mma.sync one, which shares none of its epilogues."""

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bbs():
    from paper_2308_08417_gb300 import _build, bbs as mod

    _build.build()
    return mod


@pytest.mark.parametrize("n,hidden,M,shift", [(1, 64, 64, 0), (5, 64, 64, 0), (21, 64, 192, 1), (63, 128, 512, 0),
                                              (65, 192, 576, 3), (144, 256, 4096, 0), (300, 64, 1088, 0)])
def test_training_step_tiles(bbs, n, hidden, M, shift):
    h = bbs.Handle(0)
    net = bbs.MLP(h, n, hidden=hidden, seed=3, max_batch=max(M, 1024))
    g = torch.Generator().manual_seed(n + M)
    store = 2 * M + 7
    # a store that starts `shift` elements past a 16-byte boundary
    feats = torch.zeros(store * net.in_pad + 8, dtype=torch.bfloat16)[shift:shift + store * net.in_pad]
    feats = feats.view(store, net.in_pad)
    feats[:, :3 * n] = torch.randn(store, 3 * n, generator=g).to(torch.bfloat16)
    dev = torch.zeros(store * net.in_pad + 8, dtype=torch.bfloat16, device="cuda")
    dev = dev[shift:shift + store * net.in_pad].view(store, net.in_pad)
    dev.copy_(feats)
    targets = torch.randn(store, n, generator=g).cuda()
    rows = torch.randint(0, store, (M,), generator=g, dtype=torch.int32).cuda()
    got = {}
    for kind in ("mma", "tcgen05"):
        net.set_gemm(kind)
        loss = float(net.gradients(dev, targets, rows))
        got[kind] = (loss, net.get_grads().double().cpu())
    net.check()
    # both accumulate the same BF16 products in FP32. An activation or a delta
    # next to a rounding boundary may fall to either side, 2^-8 of its size, so
    # norms of differences stay below 2^-8 of the norms.
    (l0, g0), (l1, g1) = got["mma"], got["tcgen05"]
    assert abs(l1 - l0) <= 2.0 ** -8 * l0
    o = 0
    for i, out in ((3 * n, hidden), (hidden, hidden), (hidden, hidden), (hidden, n)):
        for size in (i * out, out):
            a, b = g0[o:o + size], g1[o:o + size]
            assert (a - b).norm() <= 2.0 ** -8 * a.norm(), (o, size)
            o += size
    assert o == net.param_count

    # the step leaves the BF16 weights that its new parameters round to
    net.train_step(dev, targets, rows, 1e-3)
    X = dev[:64].clone()  # forward() takes aligned rows only
    after = net.forward(X).clone()
    net.set_params(net.get_params())
    assert torch.equal(after, net.forward(X))
