"""Refinement over ranges longer than the window (locations that enter and leave
again), single-location windows, bins with many locations and every band count;
and the same results whether a warp takes one candidate or all of a read's."""
import numpy as np
import pytest
import torch

import oracle
import synth
from _parity import dev
from test_refine_gpu import check_refine, gparams

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pp,N,radius", [
    (dict(s=2, m=2, t=1), 20, 60),
    (dict(s=4, m=1, t=4), 4, 9),
    (dict(s=3, m=8, t=1, score_mode=1), 50, 33),
    (dict(s=4, m=3, t=2), 35, 16),
    (dict(s=8, m=5, t=8), 39, 32),
])
def test_ranges(lib, pp, N, radius):
    # a quarter of the reference in short tandem repeats: bins with long chains
    ref = synth.markov_ref(4000, 0.41, 71, 0.25, 0.25)
    rd = synth.reads(ref, 24, seed=72, length=N)
    op = oracle.Params(variant=1, N=N, **pp)
    rng = np.random.default_rng(73)
    cand = np.clip(rd.true_pos[:, None] + rng.integers(-5, 6, size=(24, 3)), 0, None)
    cand[::5, 1] = -1
    cand[1, 0], cand[2, 0], cand[3, 0] = 0, len(ref) - N, len(ref) + 9
    want = oracle.refine(ref, rd.seqs, rd.offsets, cand, radius, op)
    idx = lib.rope_encode_reference(lib.Params(window_len=N), dev(ref))
    gp, gf = lib.rope_refine(idx, gparams(lib, op), dev(rd.seqs), dev(rd.offsets), dev(cand), radius)
    lib.rope_sync_status()
    check_refine(gp.cpu().numpy(), gf.cpu().numpy().astype(np.float64), *want, cand)
    idx.free()


def test_candidates_per_warp(lib):
    ref = synth.uniform_ref(50_000, 74)
    rd = synth.reads(ref, 20_000, seed=75)
    p = lib.Params(s=8, m=2, t=8, variant=1, window_len=150)
    idx = lib.rope_encode_reference(lib.Params(window_len=150), dev(ref))
    cand = dev(rd.true_pos[:, None] + np.array([[-3, 2, 700]]))
    seqs, offs = dev(rd.seqs), dev(rd.offsets)
    gp, gf = lib.rope_refine(idx, p, seqs, offs, cand, 5)
    n = 37
    hp, hf = lib.rope_refine(idx, p, seqs[:int(rd.offsets[n])], offs[:n + 1], cand[:n].contiguous(), 5)
    lib.rope_sync_status()
    assert torch.equal(gp[:n], hp) and torch.equal(gf[:n], hf)
    idx.free()
