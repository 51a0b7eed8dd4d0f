"""Host threads that call the same kernels with different shared-memory sizes
at the same time: every call launches and gives what it gives alone."""
import threading

import pytest
import torch

import synth
from _parity import dev
from paper_2603_22245_gb300 import rerank

pytestmark = pytest.mark.gpu


def _mlp(lib):
    # weight rows padded to 24 features of 500 units (52 KB), and to 32 of 310 (42 KB)
    X = [torch.rand(64, 17, device="cuda"), torch.rand(64, 32, device="cuda")]
    rr = [rerank.Reranker(17, 500, seed=1), rerank.Reranker(32, 310, seed=2)]
    return [lambda: rr[0].predict(X[0]), lambda: rr[1].predict(X[1])]


def _encode(lib):
    ref = synth.uniform_ref(50_000, 91)
    p = lib.Params(s=8, m=4, t=4, variant=1, window_len=300)
    rd = [synth.reads(ref, n, seed=92, length=300) for n in (3000, 1300)]
    a = [(dev(r.seqs), dev(r.offsets)) for r in rd]
    return [lambda: lib.rope_encode_reads(p, *a[0])[0], lambda: lib.rope_encode_reads(p, *a[1])[0]]


def _refine(lib):
    ref = synth.uniform_ref(50_000, 93)
    idx = lib.rope_encode_reference(lib.Params(window_len=150), dev(ref))
    rd = synth.reads(ref, 64, seed=94)
    s, o = dev(rd.seqs), dev(rd.offsets)
    c = torch.arange(64, device="cuda").reshape(64, 1) * 700
    p = lib.Params(s=8, m=2, t=8, variant=1, window_len=150)
    return [lambda: lib.rope_refine(idx, p, s, o, c, 300)[1], lambda: lib.rope_refine(idx, p, s, o, c, 2)[1]]


def _fp32(lib):
    ref = synth.uniform_ref(6_000, 95)
    idx = lib.rope_encode_reference(lib.Params(window_len=150), dev(ref))
    rd = synth.reads(ref, 64, seed=96)
    s, o = dev(rd.seqs), dev(rd.offsets)
    return [lambda: lib.rope_map(idx, s, o, k=32, precision="fp32")[1], lambda: lib.rope_map(idx, s, o, k=1, precision="fp32")[1]]


@pytest.mark.parametrize("calls", [_mlp, _encode, _refine, _fp32])
def test_two_sizes_at_once(lib, calls):
    fns = calls(lib)
    want = [f().clone() for f in fns]
    torch.cuda.synchronize()
    start = threading.Barrier(2)
    errors = []

    def work(f, w):
        try:
            start.wait()
            for _ in range(300):
                got = f()
            torch.cuda.synchronize()
            assert torch.equal(got, w)
        except Exception as e:  # noqa: BLE001 - reported below
            errors.append(repr(e))

    ts = [threading.Thread(target=work, args=a) for a in zip(fns, want)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    lib.rope_sync_status()
    assert not errors, errors
