"""Index build: windows that slide from a large norm into one that nearly or
wholly cancels (a homopolymer with one-letter s-mers sums all roots of unity,
and two letters half a window apart add nearly opposite phases) keep norms as
exact as any other window's."""
import numpy as np
import pytest

import oracle
from _parity import dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,stride,off", [(150, 1, 1), (10_000, 8, 3), (65_536, 64, 20)])
@pytest.mark.parametrize("m,score_mode", [(1, 0), (3, 1)])
@pytest.mark.parametrize("pair", [True, False])
def test_cancelling_windows(lib, N, stride, off, m, score_mode, pair):
    W = 3 * 64
    ref = np.full(N + (W - 1) * stride, ord("A"), dtype=np.uint8)
    ref[64 * stride:96 * stride] = ord("C")  # a chunk's first windows: large sums
    if pair:
        ref[[130 * stride, 130 * stride + N // 2 + off]] = ord("C")
    pp = dict(s=1, m=m, t=1, variant=0)
    idx = lib.rope_encode_reference(lib.Params(window_len=N, stride=stride, score_mode=score_mode, **pp), dev(ref))
    lib.rope_sync_status()
    c = oracle.windows_direct(ref, oracle.Params(N=N, stride=stride, **pp), 0, W)
    n2 = np.sum(np.abs(c) ** 2, axis=1)
    assert m > 1 or (n2 < (1e-2 if pair else 1e-9)).sum() >= 30
    want = np.where(n2 > 1e-6, 1 / np.sqrt(np.maximum(n2, 1e-6)), 0)
    # FP64 sums rounded once to FP32
    assert np.all(np.abs(idx.inv_norm().cpu().numpy()[:W] - want) <= 1.2e-7 * want)
    idx.free()
