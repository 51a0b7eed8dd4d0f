"""Wide encodings with many heads a block (a block's warps share its staged
phases, 256 locations at a time), ragged last blocks and more than one wave: a
head's row is the bits it has in a small batch, where it has a block to itself;
short heads and letters outside ACGT leave their block's other heads alone."""
import numpy as np
import pytest
import torch

import synth
from _parity import dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("s,m,t", [(8, 4, 4), (5, 5, 3), (6, 1, 6)])
@pytest.mark.parametrize("n_loc", [255, 256, 257, 520])
@pytest.mark.parametrize("n", [153, 1217, 4999])
def test_heads_of_a_block(lib, s, m, t, n_loc, n):
    N = n_loc + s - 1
    rd = synth.reads(synth.markov_ref(30_000, 0.41, 85, 0.1, 0.1), n, seed=86, length=N)
    seqs, offs = rd.seqs.copy(), rd.offsets.copy()
    short, bad = n // 2, n // 2 + 2
    offs[short + 1] -= 1  # its last letter goes to the next head, which ignores letters past N
    seqs[offs[bad] + N - 1] = ord("N")
    p = lib.Params(s=s, m=m, t=t, variant=1, window_len=N)
    f32, bf16, norms = lib.rope_encode_reads(p, dev(seqs), dev(offs))
    with pytest.raises(lib.RopeError):
        lib.rope_sync_status()
    assert not f32[[short, bad]].any() and not norms[[short, bad]].any()
    # the next head starts a letter earlier than it was made
    at = np.r_[0:6, short - 3:short + 6, n - 6:n]
    at = at[(at != short) & (at != bad)]
    parts = [seqs[offs[i]:offs[i] + N] for i in at]
    o = np.arange(len(at) + 1, dtype=np.int64) * N
    g32, g16, gn = lib.rope_encode_reads(p, dev(np.concatenate(parts)), dev(o))
    lib.rope_sync_status()
    k = torch.from_numpy(at).cuda()
    assert torch.equal(f32[k], g32) and torch.equal(bf16[k], g16) and torch.equal(norms[k], gn)
