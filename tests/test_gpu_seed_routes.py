"""Where the persistent form's seed search sends a read, from the counts at the start
of the call's scratch (reads left for more lanes, taken up there, left for the
tree): few places are answered at once, hundreds by a warp, a read with more targets than a
warp keeps goes on to the tree search, and one with more places than a warp looks at
goes there without that try."""
import numpy as np
import pytest

import paper_1505_07855_gb300 as aln
from synth import Rng, reference_iid
from test_gpu_seed import TREE, _same

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("z", [1, 4])  # 8 and 16 lanes a read
def test_routes(z):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = Rng(8, "routes")
    n, m = 200, 60
    few = reference_iid(n * 64, rng.sub("f")).reshape(n, 64)
    some, over, many = (reference_iid(m, rng.sub(x)) for x in "som")
    text = np.concatenate([few.reshape(-1)] + [np.tile(np.concatenate([unit, few[0, :9]]), copies)
                                               for unit, copies in ((some, 300), (over, 2000), (many, 20_000))])
    al = aln.Aligner(aln.Index.build(text, kmer_k=6).to_device(0))
    p = aln.Params(z=z, hit_cap=4, mode=aln.MODE_PERSISTENT, max_gapo=0)
    res, hits = al.outputs(n, 4)
    for codes, places, wide, rest in ((few[:, :m], 1, 0, 0), (np.repeat(some[None], n, 0), 300, n, 0),
                                      (np.repeat(over[None], n, 0), 2000, n, n),
                                      (np.repeat(many[None], n, 0), 20_000, 0, n)):
        d = al.upload(np.ascontiguousarray(codes).reshape(-1), np.arange(n) * m, np.full(n, m))
        scratch = torch.zeros(aln.scratch_bytes(n), dtype=torch.uint8, device="cuda")
        al.search_device(d, p, res, hits, scratch=scratch)
        got = scratch[:12].cpu().numpy().view(np.uint32)
        assert (got[0], got[2]) == (wide, rest)
        assert (res.cpu().numpy().view(aln.RES_DTYPE)["c0"][:n] == places).all()


@pytest.mark.parametrize("left", [0, 1, 5, 51, 52, 53, 399, 400])
def test_left_reads_over_the_warps(left):
    """400 reads, 13 blocks: the reads left (variants of a sequence of 20 000 copies)
    are shared out over 52 warps, whose other lanes help with their trees."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = Rng(9, "left")
    g = np.random.default_rng(left)
    n, m = 400, 60
    unit, others = reference_iid(m, rng.sub("u")), reference_iid(n * 64, rng.sub("o")).reshape(n, 64)
    copies = np.repeat(np.concatenate([unit, others[0, :9]])[None], 20_000, 0)
    copies[np.arange(0, 20_000, 9), g.integers(0, m, len(range(0, 20_000, 9)))] = 2  # and some of their variants
    al = aln.Aligner(aln.Index.build(np.concatenate([others.reshape(-1), copies.reshape(-1)]), kmer_k=6).to_device(0))
    codes = others[:, :m].copy()
    codes[:left] = unit
    codes[np.arange(left), g.integers(0, m, left)] = 1
    codes = np.ascontiguousarray(codes[g.permutation(n)]).reshape(-1)
    offsets, lens = np.arange(n) * m, np.full(n, m)
    for heavy in (0, 1):
        p = aln.Params(z=2, hit_cap=64, mode=aln.MODE_PERSISTENT, heavy_after=heavy)
        d = al.upload(codes, offsets, lens)
        res, hits = al.outputs(n, 64)
        scratch = torch.zeros(aln.scratch_bytes(n), dtype=torch.uint8, device="cuda")
        al.search_device(d, p, res, hits, scratch=scratch)
        assert int(scratch[8:12].cpu().numpy().view(np.uint32)[0]) == left
        got = res.cpu().numpy().view(aln.RES_DTYPE)[:n], hits.cpu().numpy().view(aln.HIT_DTYPE)[:n * 64].reshape(n, 64)
        p.work_limit = TREE
        _same(got, al.align(codes, offsets, lens, p), 64, left)
