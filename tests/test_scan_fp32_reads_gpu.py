"""FP32 scan with one and with two reads per thread: a read's results are the
same bits in a batch of either kind."""
import pytest
import torch

import synth
from _parity import dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pp", [dict(s=2, m=1, t=1), dict(s=4, m=2, t=1), dict(s=4, m=1, t=2), dict(s=4, m=2, t=2),
                                dict(s=4, m=4, t=2), dict(s=4, m=2, t=2, score_mode=1)])
@pytest.mark.parametrize("n", [257, 511, 513])
def test_reads_per_thread(lib, pp, n):
    ref = synth.markov_ref(30_011, 0.41, 91, 0.025, 0.025, 0.0)
    rd = synth.reads(ref, n, seed=92)
    p = lib.Params(variant=1, window_len=150, **pp)
    idx = lib.rope_encode_reference(p, dev(ref))
    e = lib.rope_encode_reads(p, dev(rd.seqs), dev(rd.offsets))
    o = dict(k=4, cand_depth=8, rescore_depth=8, precision="fp32", n_ranges=5)
    for rescore in (True, False):
        w, s = lib.rope_score_topk(idx, *e, rescore=rescore, **o)
        for a in range(0, n, 256):
            part = [v[a:a + 256].contiguous() for v in e]
            w1, s1 = lib.rope_score_topk(idx, *part, rescore=rescore, **o)
            assert torch.equal(w[a:a + 256], w1) and torch.equal(s[a:a + 256], s1)
    d = lib.rope_score_dense(idx, *e, 101, 333, precision="fp32")
    d1 = lib.rope_score_dense(idx, *[v[256:].contiguous() for v in e], 101, 333, precision="fp32")
    lib.rope_sync_status()
    assert torch.equal(d[256:], d1)
    idx.free()
