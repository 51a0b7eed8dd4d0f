"""Ragged read groups in the tensor-core scan: the read tiles of a group that
hold no reads are skipped by the threads that issue and the warps that read
their accumulators, over many consecutive window ranges of the same group."""
import pytest
import torch

import synth
from _parity import dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def case(lib):
    ref = synth.markov_ref(700_000, 0.41, 51, 0.025, 0.025, 0.0)
    rd = synth.reads(ref, 1024, seed=52)
    out = {}
    for d, m in ((64, 2), (128, 4)):
        p = lib.Params(s=4, m=m, t=2, variant=1, window_len=150)
        idx = lib.rope_encode_reference(p, dev(ref))
        out[d] = (idx, lib.rope_encode_reads(p, dev(rd.seqs), dev(rd.offsets)))
    yield out
    for idx, _ in out.values():
        idx.free()


# reads in the first tile only, one past a tile, one past a group, one past two
# groups; lists of 16 leave room for five window slots instead of six
@pytest.mark.parametrize("d,variant", [(64, 0), (64, 1), (64, 2), (128, 0)])
@pytest.mark.parametrize("n", [1, 96, 129, 257, 400, 513])
@pytest.mark.parametrize("k,sep,depth", [(4, 0, 8), (8, 150, 16)])
def test_partly_filled_groups(lib, case, d, variant, n, k, sep, depth):
    # rows do not depend on the other reads of the batch: the same rows of a
    # batch of whole groups, exactly (lists as deep as the re-scoring hold the
    # same best entries however the windows are split)
    idx, (f32, bf16, norms) = case[d]
    o = dict(k=k, sep=sep, cand_depth=depth, rescore_depth=depth)
    for reads in (n, 1024):
        lib.rope_autotune_set(idx, reads, variant, 16, k=k, sep=sep, cand_depth=depth)
    w, s = lib.rope_score_topk(idx, f32[:n], bf16[:n], norms[:n], n_ranges=171, **o)
    w1, s1 = lib.rope_score_topk(idx, f32, bf16, norms, **o)
    lib.rope_sync_status()
    assert torch.equal(w, w1[:n]) and torch.equal(s, s1[:n])


@pytest.mark.parametrize("d", [64, 128])
def test_many_items_of_a_ragged_group(lib, d):
    # 300 ranges of 16 whole groups and one of 96 reads: the blocks at the end
    # run tens of items whose second tile is empty
    ref = synth.uniform_ref(3_000_000, 53)
    rd = synth.reads(ref, 16 * 256 + 96, seed=54)
    p = lib.Params(s=4, m=2 if d == 64 else 4, t=2, variant=1, window_len=150)
    idx = lib.rope_encode_reference(p, dev(ref))
    f32, bf16, norms = lib.rope_encode_reads(p, dev(rd.seqs), dev(rd.offsets))
    w, s = lib.rope_score_topk(idx, f32, bf16, norms, k=4, n_ranges=300)
    t = slice(16 * 256, None)
    w1, s1 = lib.rope_score_topk(idx, f32[t].contiguous(), bf16[t].contiguous(), norms[t].contiguous(), k=4, n_ranges=1)
    lib.rope_sync_status()
    assert torch.equal(w[t], w1) and torch.equal(s[t], s1)
    idx.free()
