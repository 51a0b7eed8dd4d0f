"""Wide encodings (more than 128 complex entries) at the edges of a step of 32
locations and of a staged chunk of 1,024, and letters outside ACGT anywhere."""
import numpy as np
import pytest

import oracle
import synth
from _parity import dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("s,m,t", [(8, 4, 4), (5, 5, 3), (1, 8, 1)])
@pytest.mark.parametrize("n_loc", [1, 31, 32, 33, 64, 1023, 1024, 1025, 2049])
def test_head_lengths(lib, s, m, t, n_loc):
    if m * 4 ** t <= 128:
        n_loc += 6144 // m  # narrow encodings take this path where their phases exceed 48 KB
    N = n_loc + s - 1
    rd = synth.reads(synth.markov_ref(20_000, 0.41, 81, 0.1, 0.1), 19, seed=82, length=N + 3)
    op = oracle.Params(s=s, m=m, t=t, variant=1, N=N)
    f32, _, norms = lib.rope_encode_reads(lib.Params(s=s, m=m, t=t, variant=1, window_len=N), dev(rd.seqs), dev(rd.offsets))
    lib.rope_sync_status()
    D = op.dim
    f32, norms = f32.cpu().numpy(), norms.cpu().numpy()
    for i in range(rd.n):
        x = oracle.embed(rd.read(i), op)
        nrm = np.linalg.norm(x)
        assert np.all(np.abs(f32[i, :D] + 1j * f32[i, D:] - x) <= 1e-5 * nrm + 1e-6)
        assert abs(norms[i, 0] - nrm ** 2) <= 2e-5 * nrm ** 2 + 1e-5


@pytest.mark.parametrize("at", [0, 31, 32, 1030, 1199])
def test_bad_letter(lib, at):
    rd = synth.reads(synth.uniform_ref(20_000, 83), 5, seed=84, length=1200)
    seqs = rd.seqs.copy()
    seqs[rd.offsets[2] + at] = ord("N")
    p = lib.Params(s=8, m=4, t=4, variant=1, window_len=1200)
    clean, _, _ = lib.rope_encode_reads(p, dev(rd.seqs), dev(rd.offsets))
    lib.rope_sync_status()
    f32, _, norms = lib.rope_encode_reads(p, dev(seqs), dev(rd.offsets))
    with pytest.raises(lib.RopeError):
        lib.rope_sync_status()
    assert (f32[2] == 0).all() and (norms[2] == 0).all()
    others = [0, 1, 3, 4]
    assert (f32[others] == clean[others]).all()
