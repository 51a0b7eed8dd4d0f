"""The tensor-core scan with few window slots: deep candidate lists, large
strides and long windows leave shared memory for two slots and a short queue of
candidates, for one buffer of bins, or for a single slot, where each read tile has
one MMA issuer instead of two."""
import numpy as np
import pytest
import torch

import oracle
import synth
from _parity import bf16_tol, check_topk, dev, f32_tol, fp8_tol

pytestmark = pytest.mark.gpu


def _case(lib, N, stride, n, windows):
    ref = synth.markov_ref(N + stride * windows, 0.41, 71, 0.025, 0.025, 0.0)
    rd = synth.reads(ref, n, seed=72, length=N)
    p = lib.Params(s=4, m=2, t=2, variant=1, window_len=N, stride=stride)
    return ref, rd, lib.rope_encode_reference(p, dev(ref)), lib.rope_encode_reads(p, dev(rd.seqs), dev(rd.offsets))


# window slots (and queue entries): 2 (3), 1 (4), 2 (1), 2 (4, one buffer of
# bins); variant 1: 2 (4); E4M3: 2 (3)
@pytest.mark.parametrize("stride,k,variant,precision", [
    (8, 24, 0, "bf16"),
    (8, 27, 0, "bf16"),
    (4, 32, 0, "bf16"),
    (1, 32, 0, "bf16"),
    (8, 32, 1, "bf16"),
    (8, 32, 0, "fp8"),
])
@pytest.mark.parametrize("n", [1, 200, 300])  # a lone read, a ragged second tile, a ragged second group
def test_deep_lists(lib, stride, k, variant, precision, n):
    ref, rd, idx, (f32, bf16, norms) = _case(lib, 150, stride, n, 3 * 4096 + 700)
    op = oracle.Params(s=4, m=2, t=2, variant=1, N=150, stride=stride)
    ow, os_ = oracle.score_topk(ref, rd.seqs, rd.offsets, op, k=k + 1)
    lib.rope_autotune_set(idx, n, variant, 16, k=k, precision=precision)
    for n_ranges in (1, 4):  # one block with every super-tile, and a super-tile a block
        w, s = lib.rope_score_topk(idx, f32, bf16, norms, k=k, precision=precision, n_ranges=n_ranges)
        lib.rope_sync_status()
        check_topk(ref, rd, op, w.cpu().numpy(), s.cpu().numpy().astype(np.float64), ow, os_, k,
                   fp8_tol if precision == "fp8" else bf16_tol, score_tol_fn=f32_tol)
    idx.free()


# window slots (and queue entries): 2 (3), 1 (3), 1 (4); variant 1: 1 (4)
@pytest.mark.parametrize("N,stride,k,depth,variant", [
    (44_000, 8, 8, 8, 0),
    (53_000, 8, 8, 8, 0),
    (30_000, 8, 8, 16, 0),
    (46_650, 4, 32, 32, 1),
])
def test_long_windows(lib, N, stride, k, depth, variant):
    # the scan's own scores, exactly: the best of all scores as the scan without lists writes them
    _, _, idx, (f32, bf16, norms) = _case(lib, N, stride, 300, 3 * 4096 + 700)
    lib.rope_autotune_set(idx, 300, variant, 16, k=k, cand_depth=depth)
    s_all, w_all = lib.rope_score_dense(idx, f32, bf16, norms, 0, idx.n_windows, precision="bf16").sort(
        dim=1, descending=True, stable=True)
    for n_ranges in (1, 4):
        w, s = lib.rope_score_topk(idx, f32, bf16, norms, k=k, cand_depth=depth, rescore=False, n_ranges=n_ranges)
        lib.rope_sync_status()
        assert torch.equal(w, w_all[:, :k] * stride) and torch.equal(s, s_all[:, :k])
    idx.free()
