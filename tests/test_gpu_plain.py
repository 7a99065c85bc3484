"""The plain form's seed search and the tree search of the reads it leaves, in one
launch: every field of every read against the tree search alone (a work limit is
set), for batches that give a warp one read, two, a last one short, all its lanes,
and more than the device holds at once, and over the texts on which the seed
search leaves the most (repeats, tandems, a text hardly longer than a read)."""
import numpy as np
import pytest

import paper_1505_07855_gb300 as aln
from synth import Reads, Rng, reference_iid, simulate_reads
from test_gpu_seed import TREE, _reads, _same, _text

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    return t


def _both(al, reads, p, z=None):
    got = al.align(reads.codes, reads.offsets, reads.lens, p, z=z)
    p.work_limit = TREE
    tree = al.align(reads.codes, reads.offsets, reads.lens, p, z=z)
    p.work_limit = 0
    full = (tree[0]["flags"] & aln.FLAG_INCOMPLETE) != 0  # more candidates than the tree search keeps
    assert np.array_equal((got[0]["flags"] & aln.FLAG_INCOMPLETE) != 0, full)
    _same((got[0][~full], got[1][~full]), (tree[0][~full], tree[1][~full]), p.hit_cap, reads.n)
    return got


@pytest.mark.parametrize("n", [1, 3, 609, 8_001, 40_000, 130_003])
def test_batch_sizes(torch, n):
    """Half of the reads from 6000 copies of one sequence (left to the tree), half
    from between them."""
    rng = Rng(31, "plain")
    unit = reference_iid(64, rng.sub("u"))
    text = reference_iid(6000 * 100, rng.sub("t")).reshape(6000, 100)
    text[:, :64] = unit
    text = np.ascontiguousarray(text.reshape(-1))
    al = aln.Aligner(aln.Index.build(text, kmer_k=6).to_device(0))
    a = simulate_reads(text, n, 50, rng.sub("a"), z=2)
    copies = np.repeat(unit[None, 7:57], n, 0)
    g = np.random.default_rng(n)
    copies[np.arange(n), g.integers(0, 50, n)] = g.integers(0, 4, n)
    b = Reads(copies.reshape(-1), np.arange(n, dtype=np.uint64) * np.uint64(50), np.full(n, 50, np.uint16),
              np.full(n, 2, np.uint8), np.zeros(n, np.int64), np.zeros(n, np.uint8))
    reads = Reads.concat([a, b]).subset(g.permutation(2 * n)[:n])
    res, _ = _both(al, reads, aln.Params(z=1, hit_cap=4))
    if n > 1000:
        assert 0.3 < (res["c0"] + res["c1"] >= 5000).mean() < 0.8


@pytest.mark.parametrize("name", ["repeats", "tandem", "short"])
@pytest.mark.parametrize("strata", [aln.STRATA_BEST1, aln.STRATA_FULL])
def test_hard_texts(torch, name, strata):
    text = _text(name)
    al = aln.Aligner(aln.Index.build(text, kmer_k=6).to_device(0))
    lengths = tuple(x for x in (20, 33, 50, 64, 100, 150) if x + 40 < text.size)
    for z, gape, e in ((2, 2, 5), (3, 6, 0)):
        reads = _reads(text, lengths, 600, z, 70 + z)
        zz = (np.arange(reads.n) % (z + 1)).astype(np.uint8)
        for cap, zarr in ((255, None), (2, zz)):
            p = aln.Params(z=z, max_gape=gape, indel_end_skip=e, seed_len=24, seed_z=2, hit_cap=cap, strata=strata)
            _both(al, reads, p, zarr)
