"""Index build: every window's stored 1/|c| and the anchors' windows against the
FP64 oracle, at chunk edges, ragged ends, band counts that do not divide a warp
and every width of the sums."""
import numpy as np
import pytest

import oracle
import synth
from _parity import dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pp,N,stride,W", [
    (dict(s=4, m=2, t=2), 150, 1, 64 * 37 + 1),
    (dict(s=4, m=2, t=2), 150, 1, 3),
    (dict(s=1, m=1, t=1), 1, 1, 130),
    (dict(s=4, m=3, t=2), 90, 2, 64 * 11 - 1),
    (dict(s=5, m=8, t=1), 77, 3, 64 * 9 + 31),
    (dict(s=3, m=2, t=3), 64, 64, 64 * 3 + 17),
    (dict(s=8, m=4, t=2), 1031, 8, 64 * 5 + 62),
])
def test_every_window_norm(lib, pp, N, stride, W):
    L = N + (W - 1) * stride + stride - 1
    ref = synth.markov_ref(L, 0.41, 61, 0.02, 0.02, 0.0)
    op = oracle.Params(variant=1, N=N, stride=stride, **pp)
    idx = lib.rope_encode_reference(lib.Params(variant=1, window_len=N, stride=stride, **pp), dev(ref))
    lib.rope_sync_status()
    assert idx.n_windows == W
    c = oracle.windows_direct(ref, op, 0, W)
    n2 = np.sum(np.abs(c) ** 2, axis=1)
    want = np.where(n2 > 1e-6, 1 / np.sqrt(np.maximum(n2, 1e-6)), 0)
    # FP64 sums rounded once to FP32
    assert np.all(np.abs(idx.inv_norm().cpu().numpy()[:W] - want) <= 1.2e-7 * want)
    if op.dim in (4, 8, 16, 32, 64, 128):
        got = lib.rope_window_embeddings(idx, 0, W).cpu().numpy()
        at = np.arange(0, W, 64)  # the chunks' first windows are the anchors themselves
        g = got[at, :op.dim] + 1j * got[at, op.dim:]
        assert np.all(np.abs(g - c[at]) <= 1e-7 * np.sqrt(n2[at])[:, None] + 1e-7)
    idx.free()
