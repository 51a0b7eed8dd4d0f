"""The work a user has this library do, as measurable cases.

Every case is one call (or one short chain of calls) of the public Python
binding on inputs of the shapes the repository's benchmark and tests use:
mapping short reads against a reference (``rope_map``), the long-read
configuration on both strands (``rope_map_strands``), the length ladder
(``rope_ladder_map``), the FP32 plain path, building either kind of index, the
learned reranker (mapping with it, and a gradient of its training), and the
refinement of candidate loci.

Inputs are made on the GPU from the seed alone: an order-2 Markov reference at
41% GC with tandem repeats and segmental duplicates, and reads that walk it
with substitutions and short indels, as the repository's generators do.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2603_22245_gb300 import rerank
from paper_2603_22245_gb300 import rotormap as rm

# the encodings of the benchmark's workloads: d = 64 and d = 128 reals for short
# reads, 2048 reals for 20 kbp reads
ENC = {64: dict(s=4, m=2, t=2), 128: dict(s=4, m=4, t=2), 2048: dict(s=8, m=4, t=4)}
# the refinement's encoding: 4^8 bins per band, two bands
REFINE_ENC = dict(s=8, m=2, t=8)

# largest read x window work of a drawn case, in scores weighted by the dimension
MAX_MAP = 16_384 * 100_000_000


def listed():
    return [
        # one small batch against a plasmid- or BAC-sized reference: launches and latency
        dict(name="map_small", kind="map", d=64, reads=256, ref=100_000, N=150, stride=1, precision="bf16", k=8),
        # a batch of a sequencing run against a bacterial or yeast genome
        dict(name="map_mid", kind="map", d=64, reads=4096, ref=10_000_000, N=150, stride=1, precision="bf16", k=8),
        # a batch against a chromosome: the benchmark's reference, the genome-scale workloads' batch
        dict(name="map_large", kind="map", d=64, reads=16_384, ref=100_000_000, N=150, stride=1, precision="bf16", k=8),
        # the wider short-read encoding, reads of another length, a ragged batch
        dict(name="map_d128", kind="map", d=128, reads=2999, ref=5_000_011, N=250, stride=1, precision="bf16", k=8),
        # the FP32 plain path: users who want no 16-bit rounding anywhere
        dict(name="map_fp32", kind="map", d=64, reads=500, ref=2_000_000, N=150, stride=1, precision="fp32", k=8),
        # 20 kbp reads on both strands over the materialised index
        dict(name="strands_20k", kind="strands", d=2048, reads=2048, ref=30_000_000, N=20_000, stride=1250, k=8),
        # reads of 100 bp to 10 kbp, one window length of the ladder each
        dict(name="ladder", kind="ladder", d=64, reads=20_000, ref=4_000_000, n_min=100, n_max=10_000, steps=8, stride=8,
             median=2000, k=8),
        # a new reference: the on-the-fly index of the short-read encoding
        dict(name="index", kind="index", d=64, ref=10_000_000, N=150, stride=1),
        # a new reference: the materialised index of the long-read encoding
        dict(name="index_dense", kind="index_dense", d=2048, ref=10_000_000, N=20_000, stride=1250),
        # mapping with the learned reranker: 16 loci per read, the best 2 kept
        dict(name="map_rerank", kind="map_rerank", d=64, reads=4096, ref=5_000_000, N=150, stride=1, k=16, keep=2),
        # one training batch of the reranker: forward, backward, gradients
        dict(name="rerank_grad", kind="rerank_grad", batch=4096, k=16, m=2, hidden=128),
        # sliding the window around each read's two best loci under a richer encoding
        dict(name="refine", kind="refine", reads=4096, ref=5_000_000, N=150, cands=2, radius=8),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["map", "map", "map", "map", "map_fp32", "strands", "ladder", "index", "index_dense", "map_rerank",
                       "rerank_grad", "refine"])
    if kind == "map":
        d = rng.choice([64, 64, 128])
        N = rng.choice([100, 150, 150, 250, rng.randint(90, 300)])
        stride = rng.choice([1, 1, 1, 2, 4, 8])
        ref = _log(rng, 50_000, 100_000_000)
        reads = _log(rng, 64, 16_384)
        cost = 3.0 if stride > 1 else 1.0  # a strided window costs more to generate
        top = MAX_MAP * 64 // d * stride / cost
        while reads * ref > top:
            ref = max(50_000, ref // 2 + rng.randint(0, 15))
        return dict(kind="map", d=d, reads=reads, ref=ref, N=N, stride=stride, precision="bf16", k=rng.choice([8, 8, 8, 4, 1]))
    if kind == "map_fp32":
        return dict(kind="map", d=64, reads=_log(rng, 64, 1024), ref=_log(rng, 50_000, 5_000_000), N=150, stride=1,
                    precision="fp32", k=8)
    if kind == "strands":
        return dict(kind="strands", d=2048, reads=_log(rng, 64, 8192), ref=_log(rng, 1_000_000, 50_000_000), N=20_000,
                    stride=1250, k=8)
    if kind == "ladder":
        return dict(kind="ladder", d=rng.choice([64, 64, 128]), reads=_log(rng, 500, 20_000), ref=_log(rng, 500_000, 4_000_000),
                    n_min=100, n_max=10_000, steps=rng.choice([4, 8]), stride=8, median=rng.choice([300, 1000, 2000]), k=8)
    if kind == "index":
        return dict(kind="index", d=rng.choice([64, 64, 128]), ref=_log(rng, 100_000, 20_000_000), N=rng.choice([100, 150, 250]),
                    stride=rng.choice([1, 1, 2, 8]))
    if kind == "index_dense":
        return dict(kind="index_dense", d=2048, ref=_log(rng, 500_000, 20_000_000), N=20_000, stride=1250)
    if kind == "map_rerank":
        return dict(kind="map_rerank", d=64, reads=_log(rng, 64, 8192), ref=_log(rng, 500_000, 10_000_000), N=150, stride=1,
                    k=16, keep=rng.choice([1, 2, 4]))
    if kind == "rerank_grad":
        return dict(kind="rerank_grad", batch=_log(rng, 256, 16_384), k=rng.choice([8, 16]), m=rng.choice([2, 4]), hidden=128)
    return dict(kind="refine", reads=_log(rng, 64, 8192), ref=_log(rng, 100_000, 5_000_000), N=rng.choice([100, 150]),
                cands=rng.choice([1, 2, 4]), radius=rng.choice([4, 8, 16]))


# ---------------------------------------------------------------- inputs

_ACGT = (65, 67, 71, 84)


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 2654435761 % (1 << 62) + 1)
    return g


def _u(g, *shape):
    return torch.rand(*shape, generator=g, device="cuda")


def _reference(g, length):
    """Letter codes (uint8, 0..3): order-2 Markov chains side by side, then 5% repeats."""
    chains = max(1, min(65_536, length // 64))
    steps = -(-length // chains)
    w = torch.tensor([0.295, 0.205, 0.205, 0.295], device="cuda") * (0.7 + 0.6 * _u(g, 16, 4))
    w[1::4, 2] *= 0.25  # CpG is rare
    cum = torch.cumsum(w / w.sum(1, keepdim=True), 1)[:, :3].contiguous()
    out = torch.empty((steps, chains), dtype=torch.uint8, device="cuda")
    ctx = torch.randint(0, 16, (chains,), generator=g, device="cuda")
    for i in range(steps):
        nxt = (_u(g, chains, 1) > cum[ctx]).sum(1)
        out[i] = nxt
        ctx = (ctx * 4 + nxt) & 15
    ref = out.t().reshape(-1)[:length].contiguous()
    # segmental duplicates (1-8 kbp, 95-99% identical) and tandem arrays
    h = np.random.default_rng(int(torch.randint(0, 1 << 31, (1,), generator=g, device="cuda").item()))
    for _ in range(min(64, length // 160_000)):
        n = int(h.integers(1000, 8000))
        a, b = (int(h.integers(0, length - n)) for _ in range(2))
        seg = ref[a:a + n].clone()
        hit = _u(g, n) < h.uniform(0.01, 0.05)
        seg = torch.where(hit, ((seg.long() + torch.randint(1, 4, (n,), generator=g, device="cuda")) & 3).to(torch.uint8), seg)
        ref[b:b + n] = seg
        unit, n = int(h.integers(2, 51)), int(h.integers(100, 2000))
        a = int(h.integers(0, length - n - unit))
        ref[a + unit:a + unit + n] = ref[a:a + unit].repeat(n // unit + 1)[:n]
    return ref


def _letters(codes):
    return torch.tensor(_ACGT, dtype=torch.uint8, device="cuda")[codes.long()]


def _walk(g, ref, n, length, sub, indel):
    """n reads (codes [n, length]) and their true starts: substitutions, insertions, geometric deletions."""
    L = ref.numel()
    span = min(L - 1, length + length // 8 + 16)
    start = torch.randint(0, L - span, (n,), generator=g, device="cuda")
    out = torch.empty((n, length), dtype=torch.uint8, device="cuda")
    rows = max(1, (1 << 25) // length)
    for a in range(0, n, rows):
        b = min(n, a + rows)
        ev = _u(g, b - a, length)
        ins = ev < indel / 2
        dele = (ev >= indel / 2) & (ev < indel)
        skip = torch.where(dele, 1 + (torch.log(_u(g, b - a, length).clamp_min(1e-6)) / math.log(0.3)).long(), 0)
        step = torch.where(ins, 0, 1 + skip)
        off = torch.cumsum(step, 1) - step
        code = ref[(start[a:b, None] + off).clamp_(max=L - 1)].long()
        mut = _u(g, b - a, length) < sub
        rnd = torch.randint(0, 4, (b - a, length), generator=g, device="cuda")
        code = torch.where(mut, (code + 1 + rnd % 3) & 3, code)
        out[a:b] = torch.where(ins, rnd, code).to(torch.uint8)
    return out, start


def _offsets(n, length):
    return torch.arange(n + 1, dtype=torch.int64, device="cuda") * length


def _params(case):
    return rm.Params(**ENC[case["d"]], variant=1, window_len=case.get("N", 150), stride=case.get("stride", 1))


def _inputs(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    if kind == "rerank_grad":
        F = rerank.n_features(case["k"], case["m"])
        rows = 4 * case["batch"]
        top = 0.9 - 0.5 * _u(g, rows, 1)
        sc = top * torch.cumprod(1 - 0.2 * _u(g, rows, case["k"]), 1)
        X = torch.cat([sc, _u(g, rows, F - case["k"])], 1).contiguous()
        t = (0.6 * _u(g, rows)).contiguous()
        order = torch.randperm(rows, generator=g, device="cuda")[: case["batch"]].contiguous()
        return dict(X=X, t=t, order=order, F=F)
    ref = _reference(g, case["ref"])
    if kind in ("index", "index_dense"):
        return dict(ref=ref)
    if kind == "ladder":
        z = torch.randn(case["reads"], generator=g, device="cuda")
        lens = (case["median"] * torch.exp(0.7 * z)).clamp(case["n_min"], case["n_max"]).long()
        codes, _ = _walk(g, ref, case["reads"], case["n_max"], 0.032, 0.048)
        keep = torch.arange(case["n_max"], device="cuda")[None, :] < lens[:, None]
        off = torch.zeros(case["reads"] + 1, dtype=torch.int64, device="cuda")
        off[1:] = torch.cumsum(lens, 0)
        return dict(ref=ref, seqs=_letters(codes[keep]), offsets=off)
    if kind == "strands":
        codes, start = _walk(g, ref, case["reads"], case["N"], 0.05, 0.10)
        flip = torch.arange(case["reads"], device="cuda") % 2 == 1
        codes = torch.where(flip[:, None], 3 - codes.flip(1), codes).contiguous()
    elif kind == "map_rerank":
        codes, start = _walk(g, ref, case["reads"], case["N"], 0.05, 0.025)
    else:
        codes, start = _walk(g, ref, case["reads"], case["N"], 0.01, 0.005)
    return dict(ref=ref, codes=codes, start=start, seqs=_letters(codes.reshape(-1)), offsets=_offsets(*codes.shape))


def _refine_candidates(g, case, start):
    """Coarse loci around the true starts, as a stride-8 scan reports them."""
    n = start.numel()
    jit = torch.randint(-case["radius"], case["radius"] + 1, (n, case["cands"]), generator=g, device="cuda")
    cand = start[:, None] + jit
    if case["cands"] > 1:
        cand[:, 1:] = torch.randint(0, case["ref"] - case["N"], (n, case["cands"] - 1), generator=g, device="cuda")
    return cand.clamp_(0, case["ref"] - case["N"]).contiguous()


# ---------------------------------------------------------------- measured calls

def prepare(case, seed):
    kind = case["kind"]
    x = _inputs(case, seed)
    st = dict(case=case, x=x)
    if kind == "rerank_grad":
        st["rr"] = rerank.Reranker(x["F"], case["hidden"], seed=7)
        return st
    letters = _letters(x["ref"])
    if kind in ("index", "index_dense"):
        st["ref"] = letters
        st["p"] = _params(case)
    elif kind == "ladder":
        p = rm.Params(**ENC[case["d"]], variant=1, window_len=case["n_min"], stride=case["stride"])
        st["lad"] = rm.rope_ladder_create(p, letters, case["n_min"], case["n_max"], case["steps"])
    elif kind == "refine":
        st["idx"] = rm.rope_encode_reference(rm.Params(**ENC[64], variant=1, window_len=case["N"]), letters)
        st["p"] = rm.Params(**REFINE_ENC, variant=1, window_len=case["N"])
        st["cand"] = _refine_candidates(_gen(seed + 1), case, x["start"])
    elif kind == "strands":
        st["idx"] = rm.rope_encode_reference_dense(_params(case), letters)
    else:
        st["idx"] = rm.rope_encode_reference(_params(case), letters)
        if kind == "map_rerank":
            st["rr"] = rerank.Reranker(rerank.n_features(case["k"], ENC[case["d"]]["m"]), 128, seed=7)
    return st


def run(state):
    case, x = state["case"], state["x"]
    kind = case["kind"]
    if kind == "map":
        return rm.rope_map(state["idx"], x["seqs"], x["offsets"], k=case["k"], precision=case["precision"])
    if kind == "strands":
        return rm.rope_map_strands(state["idx"], x["seqs"], x["offsets"], k=case["k"])
    if kind == "ladder":
        return rm.rope_ladder_map(state["lad"], x["seqs"], x["offsets"], k=case["k"])
    if kind == "index":
        idx = rm.rope_encode_reference(state["p"], state["ref"])
        return idx.inv_norm().clone(), idx.packed().clone()
    if kind == "index_dense":
        idx = rm.rope_encode_reference_dense(state["p"], state["ref"])
        return idx.inv_norm().clone(), rm.rope_window_embeddings(idx, 0, idx.n_windows)
    if kind == "map_rerank":
        return rerank.rope_map_rerank(state["idx"], x["seqs"], x["offsets"], state["rr"], k=case["k"], keep=case["keep"])
    if kind == "rerank_grad":
        return state["rr"].grad(x["X"], x["t"], x["order"])
    return rm.rope_refine(state["idx"], state["p"], x["seqs"], x["offsets"], state["cand"], case["radius"])


# ---------------------------------------------------------------- necessary work

def _windows(case):
    return (case["ref"] - case["N"]) // case["stride"] + 1


def work(case):
    kind = case["kind"]
    if kind == "rerank_grad":
        F, H, B = rerank.n_features(case["k"], case["m"]), case["hidden"], case["batch"]
        P = H * F + 2 * H + 1
        return dict(bytes=B * (F * 4 + 4 + 8) + 2 * H * F + 6 * H + 4 * P, flops=6 * B * H * (F + 1))
    if kind in ("index", "index_dense"):
        W, D = _windows(case), case["d"] // 2
        if kind == "index":  # packed letters, 1/|c| of every window, an anchor every 64 windows
            return dict(bytes=case["ref"] * 1.25 + 4 * W + W * D // 8, flops=W * D * 12)
        # FP32 rows and the two BF16 operands, plus the inspected copy of the rows
        return dict(bytes=case["ref"] * 1.25 + 4 * W + W * 2 * D * (4 + 2 + 2 + 4), flops=W * D * 8 * (case["N"] // case["stride"]))
    n = case["reads"]
    if kind == "ladder":
        D = case["d"] // 2
        return dict(bytes=case["ref"] / 4 + n * (case["median"] + 8 + 12 * case["k"]),
                    flops=8 * D * n * (case["ref"] // case["stride"]))
    if kind == "refine":
        pos = n * case["cands"] * (2 * case["radius"] + 1)
        m = REFINE_ENC["m"]
        return dict(bytes=n * (case["N"] + 8) + n * case["cands"] * (8 + (case["N"] + 2 * case["radius"]) / 4 + 12),
                    flops=n * case["cands"] * case["N"] * 12 * m + pos * 40 * m)
    D, W = case["d"] // 2, _windows(case)
    heads = 2 * n if kind == "strands" else n
    index = W * 2 * D * 2 if kind == "strands" else case["ref"] / 4 + 4 * W
    out = n * case.get("keep", case["k"]) * 16
    return dict(bytes=n * (case["N"] + 8) + index + out, flops=8 * D * heads * W)


# ---------------------------------------------------------------- the same in 64 bits

def _tables(s, m, t, N):
    """Bin of every s-mer code (first letter most significant) and the phases [m, N - s + 1]."""
    code = np.arange(4 ** s, dtype=np.uint64)
    if s == t:
        bins = code.astype(np.int64)
    else:
        with np.errstate(over="ignore"):
            bins = ((code * np.uint64(0x9E3779B97F4A7C15)) >> np.uint64(64 - 2 * t)).astype(np.int64)
    f = [1.0] if m == 1 else [2 * k / (m - 1) + 1 for k in range(m)]
    loc = torch.arange(N - s + 1, device="cuda", dtype=torch.float64)
    ang = torch.stack([2 * math.pi * ((fk * loc / N) % 1.0) for fk in f])
    return torch.from_numpy(bins).cuda(), torch.polar(torch.ones_like(ang), ang)


def _bins(codes, s, table):
    c = torch.zeros(codes.shape[:-1] + (codes.shape[-1] - s + 1,), dtype=torch.int64, device="cuda")
    for i in range(s):
        c = c * 4 + codes[..., i:codes.shape[-1] - s + 1 + i].long()
    return table[c]


def _sum(bins, ph, nb):
    """Direct sums [n, m * nb] (complex128) of rows of bins [n, n_loc]."""
    n, m = bins.shape[0], ph.shape[0]
    out = torch.zeros((n, m * nb, 2), dtype=torch.float64, device="cuda")
    rows = max(1, (1 << 25) // bins.shape[1])
    for a in range(0, n, rows):
        b = bins[a:a + rows]
        for k in range(m):
            for c, part in enumerate((ph[k].real, ph[k].imag)):
                out[a:a + rows, k * nb:(k + 1) * nb, c].scatter_add_(1, b, part.expand(b.shape[0], -1).contiguous())
    return torch.view_as_complex(out)


def _encode(codes, enc, N):
    table, ph = _tables(enc["s"], enc["m"], enc["t"], N)
    return _sum(_bins(codes[:, :N], enc["s"], table), ph, 4 ** enc["t"])


def _encode_windows(ref, enc, N, stride):
    table, ph = _tables(enc["s"], enc["m"], enc["t"], N)
    allb = _bins(ref[None, :], enc["s"], table)[0]
    rows = allb.unfold(0, N - enc["s"] + 1, stride)
    step = max(1, (1 << 25) // rows.shape[1])
    return torch.cat([_sum(rows[a:a + step].contiguous(), ph, 4 ** enc["t"]) for a in range(0, rows.shape[0], step)])


def _unit(v):
    n = torch.linalg.vector_norm(v, dim=1, keepdim=True)
    return torch.where(n > 1e-3, v / n.clamp_min(1e-3), torch.zeros_like(v))


def _best(x, c, k):
    """The k largest fidelities of every row of x against the rows of c, best first."""
    best = torch.full((x.shape[0], k), -math.inf, dtype=torch.float64, device="cuda")
    step = max(k, (1 << 27) // x.shape[0])
    for a in range(0, c.shape[0], step):
        ip = x.conj() @ c[a:a + step].t()
        fid = ip.real ** 2 + ip.imag ** 2
        best = torch.cat([best, fid.topk(min(k, fid.shape[1]), dim=1).values], 1).topk(k, dim=1).values
    return best


def _refine_exact(case, x, cand):
    """Fidelity at the best position of every candidate's range: sums over pairs of equal s-mers."""
    s, m, N, r = REFINE_ENC["s"], REFINE_ENC["m"], case["N"], case["radius"]
    table, ph = _tables(s, m, REFINE_ENC["t"], N)
    rb = _bins(x["codes"][:, :N], s, table)
    gb = _bins(x["ref"][None, :], s, table)[0]
    last = case["ref"] - N
    n_loc = N - s + 1
    best = torch.full(cand.shape, -math.inf, dtype=torch.float64, device="cuda")

    def gram(a, b):  # per band sum over equal bins of conj(ph[l]) ph[l']
        eq = (a[:, :, None] == b[:, None, :]).to(torch.complex128)
        return sum(torch.einsum("l,nlk,k->n", ph[k].conj(), eq, ph[k]) for k in range(m))

    step = 2048
    for a in range(0, cand.shape[0], step):
        bx = rb[a:a + step]
        xx = gram(bx, bx).real
        for c in range(cand.shape[1]):
            for dlt in range(-r, r + 1):
                p = cand[a:a + step, c] + dlt
                ok = (p >= 0) & (p <= last)
                w = gb[p.clamp(0, last)[:, None] + torch.arange(n_loc, device="cuda")]
                f = gram(bx, w).abs() ** 2 / (xx * gram(w, w).real)
                best[a:a + step, c] = torch.maximum(best[a:a + step, c], torch.where(ok, f, -math.inf))
    return best


def exact(case, seed):
    kind = case["kind"]
    if kind == "rerank_grad":
        x = _inputs(case, seed)
        rr = rerank.Reranker(x["F"], case["hidden"], seed=7)
        p = torch.from_numpy(rr.params()[0]).cuda().double()
        H, F = case["hidden"], x["F"]
        W1, b1 = p[:H * F].view(H, F).bfloat16().double(), p[H * F:H * F + H].clone()
        w2, b2 = p[H * F + H:H * F + 2 * H].bfloat16().double(), p[H * F + 2 * H:].clone()
        par = [v.requires_grad_() for v in (W1, b1, w2, b2)]
        z = x["X"][x["order"]].double() @ par[0].t() + par[1]
        y = (0.5 * z * (1 + torch.erf(z / math.sqrt(2)))) @ par[2] + par[3]
        loss = ((y - x["t"][x["order"]].double()) ** 2).mean()
        g = torch.autograd.grad(loss, par)
        return torch.cat([v.reshape(-1) for v in g]), loss.detach().reshape(1)
    if kind == "map" and case["reads"] * _windows(case) <= 1_500_000_000:
        x = _inputs(case, seed)
        enc = ENC[case["d"]]
        c = _unit(_encode_windows(x["ref"], enc, case["N"], case["stride"]))
        return None, _best(_unit(_encode(x["codes"], enc, case["N"])), c, case["k"])
    if kind == "strands" and case["reads"] * _windows(case) <= 60_000_000:
        x = _inputs(case, seed)
        enc = ENC[case["d"]]
        c = _unit(_encode_windows(x["ref"], enc, case["N"], case["stride"]))
        both = torch.cat([x["codes"], 3 - x["codes"].flip(1)])
        f = _best(_unit(_encode(both, enc, case["N"])), c, case["k"])
        n = case["reads"]
        return None, torch.cat([f[:n], f[n:]], 1).topk(case["k"], dim=1).values, None
    if kind in ("index", "index_dense"):
        x = _inputs(case, seed)
        enc = ENC[case["d"]]
        if kind == "index_dense":
            c = _encode_windows(x["ref"], enc, case["N"], case["stride"])
            inv = 1 / torch.linalg.vector_norm(c, dim=1)
            return inv, torch.cat([c.real, c.imag], 1)
        W, inv = _windows(case), []
        for a in range(0, W, 1 << 20):
            b = min(W, a + (1 << 20))
            c = _encode_windows(x["ref"][a * case["stride"]:(b - 1) * case["stride"] + case["N"]], enc, case["N"], case["stride"])
            n2 = (c.real ** 2 + c.imag ** 2).sum(1)
            inv.append(torch.where(n2 > 1e-6, n2.clamp_min(1e-6).rsqrt(), torch.zeros_like(n2)))
        return torch.cat(inv), None
    if kind == "refine" and case["reads"] * case["cands"] * (2 * case["radius"] + 1) <= 300_000:
        x = _inputs(case, seed)
        cand = _refine_candidates(_gen(seed + 1), case, x["start"])
        return None, _refine_exact(case, x, cand)
    return None
