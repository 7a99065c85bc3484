"""The calls a user of this library makes, as cases that can be timed and compared.

A reference is indexed once (fm_index_build_gpu, prefix-trie depth 10) and held on
the GPU; batches of reads are then searched on it, their hits compacted, located
and paired, through the Python binding.  The references follow the recipes of
the repository's workloads:

  iid     i.i.d. ACGT (the 1 Mbp text of the tiny36 workload)
  markov  order-3 Markov text, 41 % GC, 5 % copies of 50 repeat families (chr100)
  human   i.i.d. text, 45 % copies of 500 repeat families, 1 % N (human_*)

They are drawn on the GPU from a fixed seed (a program keeps its reference); the
reads come from the case's seed, with substitutions, short indels, N bases and
both strands, as those workloads have them.
"""
import collections

import numpy as np
import torch

import paper_1505_07855_gb300 as aln

DEVICE = 0
KMER_K = 10
TEXT_SEED = 20150507
MAX_WIDTH = 16

# Search limits of the repository's workloads, and z = min(6, ceil(0.04 len)) by length.
GAPS = dict(max_gapo=1, max_gape=2, seed_len=0, seed_z=0, indel_end_skip=5)
LIMITS = {
    "iid": dict(z=2, **GAPS),
    "markov": dict(z=4, max_gapo=1, max_gape=6, seed_len=32, seed_z=2, indel_end_skip=5),
    "human": dict(z=4, **GAPS),
}
MIXED_LENS = (36, 50, 76, 100, 150, 250)
STRATA = {"best1": aln.STRATA_BEST1, "full": aln.STRATA_FULL, "score": aln.STRATA_SCORE}
# (substitution rate at the 5' end, at the 3' end, indel rate per base, longest indel, reads with an N)
ERRORS = {"iid": (0.01, 0.01, 0.0005, 1, 0.02), "markov": (0.005, 0.02, 0.0002, 3, 0.0),
          "human": (0.01, 0.01, 0.0005, 1, 0.02)}


def listed():
    return [
        # One small request as an interactive caller sends it: the latency of a call.
        dict(name="search_64x36", op="search", text="iid", text_len=1_000_000, reads=64, len=36, z=2, strata="best1",
             mode="persistent", hit_cap=32),
        # The tiny36 workload captured in a CUDA graph and replayed.
        dict(name="graph_10kx36", op="graph", text="iid", text_len=1_000_000, reads=10_000, len=36, z=2,
             strata="best1", mode="persistent", hit_cap=32),
        # The chr100 benchmark batch.
        dict(name="search_1Mx100", op="search", text="markov", text_len=100_000_000, reads=1_000_000, len=100, z=4,
             strata="best1", mode="persistent", hit_cap=32),
        # Params' default mode: one thread per read, one launch.
        dict(name="plain_100kx100", op="search", text="markov", text_len=100_000_000, reads=100_000, len=100, z=4,
             strata="best1", mode="plain", hit_cap=32),
        # Every hit within z, on short reads of a ragged length.
        dict(name="full_30kx51", op="search", text="markov", text_len=100_000_000, reads=30_011, len=51, z=2,
             strata="full", mode="persistent", hit_cap=16),
        # Hits ranked by penalty score.
        dict(name="score_20kx76", op="search", text="markov", text_len=100_000_000, reads=20_000, len=76, z=3,
             strata="score", mode="persistent", hit_cap=16),
        # Host arrays in, host arrays out: the convenience call, packing and copies included.
        dict(name="align_100kx100", op="align", text="markov", text_len=100_000_000, reads=100_000, len=100, z=4,
             strata="best1", mode="persistent", hit_cap=32),
        # Requests of 1 to 20 000 reads of 50 to 250 bp through the serving loop.
        dict(name="serve_16", op="serve", text="markov", text_len=100_000_000, reads=40_000, requests=16, len=0, z=6,
             strata="best1", mode="persistent", hit_cap=8),
        # A reference brought up: its index built on the GPU, uploaded, and a first batch aligned and located.
        dict(name="index_100M", op="index", text="markov", text_len=100_000_000, reads=2_000, len=100, z=4,
             strata="best1", mode="persistent", hit_cap=16),
        # Mixed lengths of 36 to 250 bp with z by length on a human-sized reference.
        dict(name="mixed_400k", op="search", text="human", text_len=3_100_000_000, reads=400_000, len=0, z=6,
             strata="best1", mode="persistent", hit_cap=32),
        # Mates of 2 x 100 bp on it: search, compaction, positions and pairing.
        dict(name="pairs_300k", op="pairs", text="human", text_len=3_100_000_000, reads=300_000, len=100, z=4,
             strata="best1", mode="persistent", hit_cap=32),
        # What follows a search: hits compacted and located.
        dict(name="positions_500k", op="positions", text="human", text_len=3_100_000_000, reads=500_000, len=100, z=4,
             strata="best1", mode="persistent", hit_cap=32),
    ]


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    op = rng.choice(["search"] * 6 + ["plain", "graph", "align", "serve", "index", "pairs", "positions"])
    text = rng.choice(["iid", "markov", "markov", "human"])
    if op == "index":
        text = rng.choice(["iid", "markov"])
        return dict(op=op, text=text, text_len=_log(rng, 1_000_000, 100_000_000), reads=_log(rng, 200, 2_000),
                    len=rng.randint(30, 150), z=rng.randint(1, 3), strata="best1", mode="persistent", hit_cap=16)
    if op in ("pairs", "positions"):
        text = "human"
    if op in ("plain", "serve"):
        text = rng.choice(["iid", "markov"])
    c = dict(op="search" if op == "plain" else op, text=text, mode="plain" if op == "plain" else "persistent",
             hit_cap=rng.choice([4, 8, 16, 32, 32, 64]),
             text_len={"iid": _log(rng, 300_000, 30_000_000), "markov": 100_000_000, "human": 3_100_000_000}[text])
    if op == "serve":
        return dict(c, reads=_log(rng, 2_000, 40_000), requests=rng.randint(3, 24), len=0, z=6, strata="best1",
                    hit_cap=8)
    if op == "pairs":
        return dict(c, reads=2 * _log(rng, 1_000, 150_000), len=rng.randint(50, 125), z=rng.randint(2, 4),
                    strata="best1")
    if op == "positions":
        return dict(c, reads=_log(rng, 10_000, 500_000), len=rng.randint(50, 125), z=rng.randint(2, 4), strata="best1")
    strata = "best1" if c["mode"] == "plain" else rng.choice(["best1"] * 5 + ["full", "score"])
    if strata != "best1":
        return dict(c, reads=_log(rng, 100, 20_000), len=rng.randint(40, 110), z=rng.randint(1, 2), strata=strata,
                    text="markov", text_len=100_000_000)
    if rng.random() < 0.3:  # mixed lengths, z by length
        return dict(c, reads=_log(rng, 100, {"iid": 100_000, "markov": 200_000, "human": 300_000}[text]
                                  if c["mode"] != "plain" else 20_000), len=0, z=6, strata=strata)
    length = rng.randint(32, 151)
    z = rng.randint(1, min(5, (4 * length + 99) // 100 + 1))
    most = 1_000_000 if z <= 3 and c["mode"] != "plain" and text != "human" else 100_000
    return dict(c, reads=_log(rng, 16, most), len=length, z=z, strata=strata)


# ------------------------------------------------------------------ references


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed & 0x7FFFFFFFFFFFFFFF)
    return g


def _randint(g, lo, hi, size, dtype=torch.int64):
    return torch.randint(lo, hi, size, generator=g, device="cuda", dtype=dtype)


def _markov(n, g):
    """Order-3 chains of 1024 bases, the transition table drawn around 41 % GC."""
    base = torch.tensor([0.295, 0.205, 0.205, 0.295], device="cuda", dtype=torch.float64)
    t = base * (0.8 + 0.4 * torch.rand(64, 4, generator=g, device="cuda", dtype=torch.float64))
    cum = torch.cumsum(t / t.sum(1, keepdim=True), 1)[:, :3].contiguous()
    seg = 1024
    k = (n + seg - 1) // seg
    out = torch.empty(seg, k, device="cuda", dtype=torch.uint8)
    ctx = _randint(g, 0, 64, (k,))
    for j in range(seg):
        u = torch.rand(k, 1, generator=g, device="cuda", dtype=torch.float64)
        b = (u >= cum[ctx]).sum(1)
        out[j] = b
        ctx = ((ctx << 2) | b) & 63
    return out.t().contiguous().reshape(-1)[:n].clone()


def _repeats(text, g, frac, families):
    """Copies of random families (300-6000 bp, 2-15 % substitutions, either
    orientation), one after the other with random gaps between them."""
    n = text.numel()
    flen = _randint(g, 300, 6001, (families,))
    foff = torch.cumsum(flen, 0) - flen
    fam = _randint(g, 0, 4, (int(flen.sum()),), torch.uint8)
    copies = max(1, int(frac * n / 3150))
    f = _randint(g, 0, families, (copies,))
    f = f[torch.cumsum(flen[f], 0) <= int(0.9 * n)]
    copies = f.numel()
    lens = flen[f]
    w = _randint(g, 1, 65536, (copies + 1,))
    gap = w * (n - int(lens.sum())) // int(w.sum())
    start = torch.cumsum(gap[:-1] + lens, 0) - lens
    div = 0.02 + 0.13 * torch.rand(copies, generator=g, device="cuda")
    flip = _randint(g, 0, 2, (copies,))
    step = 16384
    for c0 in range(0, copies, step):
        c1 = min(copies, c0 + step)
        L = lens[c0:c1]
        who = torch.repeat_interleave(torch.arange(c0, c1, device="cuda"), L)
        j = torch.arange(who.numel(), device="cuda") - torch.repeat_interleave(torch.cumsum(L, 0) - L, L)
        back = flip[who] == 1
        src = foff[f[who]] + torch.where(back, lens[who] - 1 - j, j)
        b = fam[src].to(torch.int64)
        b = torch.where(back, 3 - b, b)
        hit = torch.rand(who.numel(), generator=g, device="cuda") < div[who]
        b = torch.where(hit, (b + _randint(g, 1, 4, (who.numel(),))) & 3, b)
        text[start[who] + j] = b.to(torch.uint8)


def _n_runs(text, g, frac):
    n = text.numel()
    runs = max(1, int(frac * n / 5050))
    lens = _randint(g, 100, 10_001, (runs,))
    pos = _randint(g, 0, max(1, n - 10_000), (runs,))
    at = torch.repeat_interleave(pos, lens) + torch.arange(int(lens.sum()), device="cuda") \
        - torch.repeat_interleave(torch.cumsum(lens, 0) - lens, lens)
    text[at] = 4


def _text(kind, n, seed):
    g = _gen(seed)
    if kind == "markov":
        text = _markov(n, g)
        _repeats(text, g, 0.05, 50)
    else:
        text = _randint(g, 0, 4, (n,), torch.uint8)
        if kind == "human":
            _repeats(text, g, 0.45, 500)
            _n_runs(text, g, 0.01)
    return text


_references = collections.OrderedDict()  # (kind, length) -> (text on the GPU, device index); the last three


def _reference(kind, n):
    key = (kind, n)
    if key not in _references:
        text = _text(kind, n, TEXT_SEED)
        dix = aln.Index.build(text.cpu().numpy(), kmer_k=KMER_K, device=DEVICE).to_device(DEVICE)
        _references[key] = (text, dix)
        while len(_references) > 3:
            _references.popitem(last=False)
        torch.cuda.empty_cache()
    _references.move_to_end(key)
    return _references[key]


# ------------------------------------------------------------------ reads


def _simulate(text, lens, g, errors, start=None, rev=None):
    """Reads of the given lengths (a tensor) as codes back to back, in 5' to 3' order."""
    sub0, sub1, indel, longest, n_frac = errors
    n, r = text.numel(), lens.numel()
    top = int(lens.max())
    pad = 4 * longest + 8
    if start is None:
        start = (torch.rand(r, generator=g, device="cuda", dtype=torch.float64) * (n - lens - 2 * pad)).long() + pad
        rev = _randint(g, 0, 2, (r,))
    parts = []
    j = torch.arange(top, device="cuda")
    for c0 in range(0, r, 1 << 18):
        L, s, v = lens[c0:c0 + (1 << 18), None], start[c0:c0 + (1 << 18), None], rev[c0:c0 + (1 << 18), None]
        k = L.numel()
        u = torch.rand(k, top, generator=g, device="cuda")
        size = _randint(g, 1, longest + 1, (k, top))
        ins = u < indel / 2
        gone = (u >= indel / 2) & (u < indel)
        use = torch.where(ins, 0, 1) + torch.where(gone, size, 0)  # text bases used up to this read base
        src = torch.cumsum(use, 1) - 1
        pos = torch.where(v == 1, s + L - 1 - src, s + src).clamp_(0, n - 1)
        b = text[pos].to(torch.int64)
        b = torch.where((v == 1) & (b < 4), 3 - b, b)
        other = _randint(g, 0, 4, (k, top))
        b = torch.where(ins, other, b)
        rate = sub0 + (sub1 - sub0) * j / (L - 1).clamp(min=1)
        hit = (torch.rand(k, top, generator=g, device="cuda") < rate) & (b < 4)
        b = torch.where(hit, (b + 1 + other % 3) & 3, b)
        if n_frac:
            at = (torch.rand(k, 1, generator=g, device="cuda") * L).long()
            b = torch.where((torch.rand(k, 1, generator=g, device="cuda") < n_frac) & (j == at), 4, b)
        parts.append(b[j < L].to(torch.uint8))
    return torch.cat(parts).cpu().numpy()


def _z_of(lens):
    return ((4 * lens + 99) // 100).clamp(max=6)


def _batch(case, seed, text):
    """Host reads of a case: codes, offsets, lens and per-read z (or None)."""
    g = _gen(seed * 2654435761 + 97)
    n = case["reads"]
    errors = ERRORS[case["text"]]
    z = None
    if case["op"] == "pairs":
        length = case["len"]
        frag = (500 + 50 * torch.randn(n // 2, generator=g, device="cuda")).round().long().clamp(min=max(200, length))
        at = (torch.rand(n // 2, generator=g, device="cuda", dtype=torch.float64) * (text.numel() - 2000)).long() + 100
        flip = _randint(g, 0, 2, (n // 2,))
        lost = torch.rand(n // 2, generator=g, device="cuda") < 0.001  # mates of unrelated places
        far = (torch.rand(n // 2, generator=g, device="cuda", dtype=torch.float64) * (text.numel() - 2000)).long() + 100
        tail = torch.where(lost, far, at + frag - length)
        start = torch.stack([torch.where(flip == 1, tail, at), torch.where(flip == 1, at, tail)], 1).reshape(-1)
        rev = torch.stack([flip, 1 - flip], 1).reshape(-1)
        lens = torch.full((n,), length, device="cuda", dtype=torch.int64)
        codes = _simulate(text, lens, g, errors, start, rev)
    else:
        if case["len"]:
            lens = torch.full((n,), case["len"], device="cuda", dtype=torch.int64)
        elif case["op"] == "serve":
            lens = _randint(g, 50, 251, (n,))
        else:
            lens = torch.tensor(MIXED_LENS, device="cuda")[_randint(g, 0, len(MIXED_LENS), (n,))]
        if not case["len"]:
            z = _z_of(lens).to(torch.uint8).cpu().numpy()
        codes = _simulate(text, lens, g, errors)
    offsets = (torch.cumsum(lens, 0) - lens).cpu().numpy().astype(np.uint64)
    return codes, offsets, lens.cpu().numpy().astype(np.uint16), z


def _params(case):
    lim = dict(LIMITS[case["text"]] if case["len"] else GAPS, z=case["z"])
    return aln.Params(**lim, hit_cap=case["hit_cap"], strata=STRATA[case["strata"]],
                      mode=aln.MODE_PLAIN if case["mode"] == "plain" else aln.MODE_PERSISTENT)


# ------------------------------------------------------------------ the cases' calls


def prepare(case, seed):
    op, p = case["op"], _params(case)
    if op == "index":
        text = _text(case["text"], case["text_len"], seed + 1)
        return dict(op=op, p=p, text=text.cpu().numpy(), batch=_batch(case, seed, text))
    text, dix = _reference(case["text"], case["text_len"])
    codes, offsets, lens, z = _batch(case, seed, text)
    s = dict(op=op, p=p, dix=dix, n=case["reads"], cap=case["hit_cap"])
    if op == "serve":
        cut = np.random.RandomState(seed % (1 << 31)).exponential(size=case["requests"]) ** 2  # few large, many small
        ends = np.minimum(np.cumsum(np.maximum(1, cut / cut.sum() * s["n"])).astype(np.int64), s["n"])
        ends[-1] = s["n"]
        s["requests"] = []
        for a, b in zip(np.concatenate([[0], ends[:-1]]), ends):
            if b > a:
                o = int(offsets[a])
                e = int(offsets[b - 1]) + int(lens[b - 1])
                s["requests"].append((codes[o:e], offsets[a:b] - np.uint64(o), lens[a:b], z[a:b]))
        s["server"] = aln.Server(dix, p, n_slots=2, max_batch_reads=1 << 15, device_mem_budget=1 << 30)
        return s
    al = s["al"] = aln.Aligner(dix)
    if op == "align":
        s["host"] = (codes, offsets, lens)
        s["z"] = z
        return s
    d = s["d"] = al.upload(codes, offsets, lens, z)
    s["res"], s["hits"] = al.outputs(s["n"], s["cap"])
    s["res"].zero_()
    s["hits"].zero_()
    if op == "graph":
        s["graph"] = al.capture(d, p, s["res"], s["hits"])
    elif op == "positions":
        al.search_device(d, p, s["res"], s["hits"])
        s["off"] = torch.zeros(s["n"] + 1, dtype=torch.int32, device="cuda")
        s["dense"] = torch.zeros(s["n"] * aln.HIT_DTYPE.itemsize, dtype=torch.uint8, device="cuda")  # room for one a read
        s["scratch"] = al.compact_scratch(s["n"])
        s["pos"] = torch.zeros(s["n"] * MAX_WIDTH, dtype=torch.int64, device="cuda")
        s["npos"] = torch.zeros(s["n"], dtype=torch.int32, device="cuda")
    return s


def _words(a):
    """A record array as 32-bit words."""
    return np.ascontiguousarray(a).view(np.int32)


def _written(res, hits):
    """The hits a search wrote, each read's slots past them cleared."""
    hits[np.arange(hits.shape[1])[None, :] >= res["n_hits"][:, None]] = 0
    return hits


def run(s):
    op, p = s["op"], s["p"]
    if op == "index":
        idx = aln.Index.build(s["text"], kmer_k=KMER_K, device=DEVICE)
        al = aln.Aligner(idx.to_device(DEVICE))
        codes, offsets, lens, z = s["batch"]
        res, hits = al.align(codes, offsets, lens, p, z=z)
        hits = _written(res, hits)
        pos, npos = al.positions(hits[:, 0], MAX_WIDTH)  # the best hit of each read
        return {"info": idx.info(), "reads": _words(res), "hits": _words(hits), "npos": npos, "pos": pos}
    if op == "serve":
        ids = [s["server"].submit(*q) for q in s["requests"]]
        out = []
        for i, q in zip(ids, s["requests"]):
            res, hits, _ = s["server"].poll(i, q[2].size)
            out.append((_words(res), _words(_written(res, hits))))
        return {"reads": np.concatenate([a for a, _ in out]), "hits": np.concatenate([b for _, b in out])}
    al = s["al"]
    if op == "align":
        res, hits = al.align(*s["host"], p, z=s["z"])
        return {"reads": _words(res), "hits": _words(_written(res, hits))}
    if op == "positions":
        al.compact(s["res"], s["hits"], s["n"], s["cap"], s["off"], s["dense"], s["scratch"])
        s["dix"].sa_to_pos(s["dense"], s["n"], MAX_WIDTH, s["pos"], s["npos"])
        return {"offsets": s["off"], "hits": s["dense"].view(torch.int32), "pos": s["pos"], "npos": s["npos"]}
    if op == "graph":
        s["graph"].replay()
    else:
        al.search_device(s["d"], p, s["res"], s["hits"])
    out = {"reads": s["res"].view(torch.int32), "hits": s["hits"].view(torch.int32)}
    if op == "pairs":
        pairs, stats = al.pair(s["res"], s["n"], s["cap"], s["hits"], MAX_WIDTH)
        out.update(pairs=_words(pairs), stats=stats)
    return out


def work(case):
    """Reads in (2-bit bases, N bits, offsets, lengths), results and about one hit
    per read out, and the index rows that a read's own bases lead to: one 64-byte
    Occ block per base and strand, or the whole index once if that is less."""
    n, m = case["reads"], case["len"] or (150 if case["op"] == "serve" else 110)
    index = case["text_len"] * 2 * 64 // 192
    if case["op"] == "positions":  # compacted hits out and read again, a sampled-SA word and a position each
        return {"bytes": n * (12 + 16 + 16 + 4 + 4 + 8 * MAX_WIDTH + 4 + 64), "flops": 0}
    b = n * (m * 3 // 8 + 8 + 2 + 12 + 16) + min(n * m * 2 * 64, index)
    if case["op"] == "index":  # the text in, the image out and onto the device
        b += case["text_len"] + 2 * (index + 2 * case["text_len"] * 4 // 32 + 2 * 8 * 4 ** (KMER_K + 1) // 3)
    if case["op"] == "pairs":
        b += n * (16 + 4 + 8 + 16)
    return {"bytes": b, "flops": 0}


def exact(case, seed):
    """Every output is a whole number, held to equality; none is a rounded value."""
    return None
