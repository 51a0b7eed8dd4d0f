"""Refinement: positions whose fidelities differ by no more than the rounding of
their FP64 sums are ties, which go to the lower one. Half a window further on
every phase is exactly negated, so where a read shares few s-mers with a range
without repeated s-mers, two positions N / 2 apart have the same sums."""
import numpy as np
import pytest

import oracle
import synth
from _parity import dev

pytestmark = pytest.mark.gpu


def test_ties_go_to_the_lower(lib):
    n, N, radius = 1500, 150, 80
    ref = synth.uniform_ref(40_011, 7)
    rd = synth.reads(ref, n, seed=3, length=N)
    cand = np.random.default_rng(11).integers(radius, len(ref) - N - radius, (n, 2))  # unrelated loci
    p = dict(s=8, m=2, t=8, variant=1)
    idx = lib.rope_encode_reference(lib.Params(window_len=N), dev(ref))
    pos, _ = lib.rope_refine(idx, lib.Params(window_len=N, **p), dev(rd.seqs), dev(rd.offsets), dev(cand), radius)
    lib.rope_sync_status()
    pos = pos.cpu().numpy()
    # the candidates whose range holds every s-mer once
    code = sum((np.frombuffer(ref, np.uint8) >> 1 & 3)[i:len(ref) - 7 + i].astype(np.int64) << (2 * i) for i in range(8))
    smers = code[(cand - radius)[:, :, None] + np.arange(2 * radius + N - 7)]
    once = np.all(np.diff(np.sort(smers, axis=2), axis=2) > 0, axis=2)
    r, c = np.nonzero(once & (pos - N // 2 >= cand - radius))
    op = oracle.Params(N=N, **p)
    at, below = pos[r, c], pos[r, c] - N // 2
    f = oracle.score_pairs(ref, rd.seqs, rd.offsets, np.r_[r, r], np.r_[at, below], op).reshape(2, -1)
    assert len(r) > 100
    tie = f[1] >= f[0] * (1 - 1e-13)
    assert not tie.any(), f"{tie.sum()} of {len(r)}"
    idx.free()
