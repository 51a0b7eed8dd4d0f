"""Reranker network over feature counts (every padded width and its edges),
hidden units that leave a group of eight unfilled, and batches at the edges of a
tile of 32 samples and of the blocks that share a batch."""
import numpy as np
import pytest
import torch

import oracle
from test_rerank_gpu import _random_net

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rr_mod(lib):
    from paper_2603_22245_gb300 import rerank

    return rerank


@pytest.mark.parametrize("F,H", [(1, 1), (8, 7), (9, 8), (16, 130), (17, 9), (24, 128), (25, 16), (32, 200)])
@pytest.mark.parametrize("B", [1, 31, 32, 33, 255, 257, 1500])
def test_shapes(rr_mod, F, H, B):
    rr, net = _random_net(rr_mod, F, H, seed=F)
    rng = np.random.default_rng(B)
    X = rng.normal(size=(B + 5, F)).astype(np.float32)
    t = rng.uniform(0, 0.3, size=B + 5).astype(np.float32)
    sel = rng.permutation(B + 5)[:B].astype(np.int64)
    Xd, td, sd = torch.from_numpy(X).cuda(), torch.from_numpy(t).cuda(), torch.from_numpy(sel).cuda()
    y = rr.predict(Xd).cpu().numpy().astype(np.float64)
    assert np.allclose(y, net.forward(X.astype(np.float64)), rtol=1e-5, atol=1e-5)
    for idx in (sd, None):
        g, loss = rr.grad(Xd, td, idx)
        rows = sel if idx is not None else np.arange(B + 5)
        l64, gW1, gb1, gw2, gb2 = net.grad(X[rows].astype(np.float64), t[rows].astype(np.float64))
        want = np.concatenate([gW1.ravel(), gb1, gw2, [gb2]])
        assert float(loss.item()) == pytest.approx(l64, rel=1e-4)
        assert np.abs(g.cpu().numpy() - want).max() <= 1e-4 * np.abs(want).max()
    # a second pass gives the same bits
    g2, loss2 = rr.grad(Xd, td, None)
    assert torch.equal(g, g2) and torch.equal(loss, loss2)
    rr.free()
