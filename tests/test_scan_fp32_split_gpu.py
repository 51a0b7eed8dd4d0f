"""FP32 scan over enough windows for two reads per thread: whole, ragged and odd
numbers of groups of 256 reads give the bits of small batches, which take one."""
import pytest
import torch

import synth
from _parity import dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def case(lib):
    ref = synth.markov_ref(2_000_011, 0.41, 95, 0.025, 0.025, 0.0)
    rd = synth.reads(ref, 2600, seed=96)
    p = lib.Params(s=4, m=2, t=2, variant=1, window_len=150)
    idx = lib.rope_encode_reference(p, dev(ref))
    yield idx, lib.rope_encode_reads(p, dev(rd.seqs), dev(rd.offsets))
    idx.free()


# groups of 256: two, three (one read per thread), four, five (one), eleven
@pytest.mark.parametrize("n", [257, 512, 513, 1000, 1025, 2600])
def test_topk(lib, case, n):
    # lists as deep as what the merge takes hold the same best entries however
    # the windows are split
    idx, e = case
    o = dict(k=4, cand_depth=8, precision="fp32")
    w, s = lib.rope_score_topk(idx, *[v[:n] for v in e], **o)
    for a in range(0, n, 256):
        w1, s1 = lib.rope_score_topk(idx, *[v[a:min(a + 256, n)].contiguous() for v in e], **o)
        lib.rope_sync_status()
        assert torch.equal(w[a:a + 256], w1) and torch.equal(s[a:a + 256], s1)


@pytest.mark.parametrize("n", [300, 513, 1000])
def test_dense(lib, case, n):
    idx, e = case
    d = lib.rope_score_dense(idx, *[v[:n] for v in e], 1_001, 180_000, precision="fp32")
    for a in range(0, n, 256):
        d1 = lib.rope_score_dense(idx, *[v[a:min(a + 256, n)].contiguous() for v in e], 1_001, 180_000, precision="fp32")
        lib.rope_sync_status()
        assert torch.equal(d[a:a + 256], d1)
