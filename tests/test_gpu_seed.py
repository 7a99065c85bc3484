"""The seed search (reads answered from the places of their error-free parts)
against the tree search, which the oracle tests pin: a search whose work limit
is set runs the tree search alone.  Every field of every read and hit, over
texts with unique, repeated, tandem and low-complexity sequence, reads at both
ends of the text, lengths from 1 to 255, N bases, every z, gap, seed and
end-window setting the seed search takes, and the three strata."""
import numpy as np
import pytest

import oracle
import paper_1505_07855_gb300 as aln
from parity_util import HIT_FIELDS, compare, oracle_align
from synth import Reads, Rng, reference_iid, simulate_reads

pytestmark = pytest.mark.gpu
TREE = 1 << 24  # the default work limit, given explicitly


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    return t


def _text(name):
    rng = Rng(123, name)
    if name == "iid":
        return reference_iid(60_000 + 77, rng.sub("t"))
    if name == "repeats":  # copies of one family, exact and diverged, in both orientations
        t = reference_iid(50_000, rng.sub("t"))
        fam = reference_iid(700, rng.sub("f"))
        for i in range(40):
            c = fam.copy()
            hit = rng.sub(f"d{i}").u64(700) % np.uint64(100) < np.uint64(i % 5)
            c[hit] = (c[hit] + 1) & 3
            if i % 3 == 0:
                c = 3 - c[::-1]
            t[1000 + 1200 * i:1700 + 1200 * i] = c
        return t
    if name == "tandem":  # units of 3 and 17 bases repeated, homopolymers, between random stretches
        t = reference_iid(30_000, rng.sub("t"))
        t[2000:2300] = np.tile(t[:3], 100)
        t[9000:9000 + 17 * 30] = np.tile(t[100:117], 30)
        t[15_000:15_060] = 0
        t[20_000:20_500] = 2
        return t
    return reference_iid(300, rng.sub("t"))  # "short": little more than a read


def _reads(text, lengths, n, z, seed):
    rng = Rng(seed, "reads")
    r = simulate_reads(text, n, lengths, rng, sub_rate=(0.01, 0.03), indel_rate=0.006, indel_lens=(1, 2, 3),
                       n_frac=0.1, z=z)
    parts = [r]
    for m in sorted(set(int(x) for x in np.atleast_1d(lengths))):  # the text's two ends, both strands
        m = min(m, text.size)
        for piece in (text[:m], text[-m:]):
            for rev in (0, 1):
                c = (3 - piece[::-1]) if rev else piece
                c = c.astype(np.uint8).copy()
                for edit in (c, np.delete(c, m // 2), np.insert(c, m // 2, 1)[:255]):
                    parts.append(Reads(edit, np.zeros(1, np.uint64), np.array([edit.size], np.uint16),
                                       np.array([z], np.uint8), np.zeros(1, np.int64), np.zeros(1, np.uint8)))
    return Reads.concat([p for p in parts if p.codes.size])


def _same(a, b, cap, what):
    ra, ha = a
    rb, hb = b
    bad = np.nonzero(ra != rb)[0]
    assert bad.size == 0, (what, bad[:5], ra[bad[:5]], rb[bad[:5]])
    valid = np.arange(cap)[None, :] < ra["n_hits"][:, None]
    for f in HIT_FIELDS:
        bad = np.argwhere(np.where(valid, ha[f], 0) != np.where(valid, hb[f], 0))
        assert bad.size == 0, (what, f, bad[0], ha[bad[0][0]][:4], hb[bad[0][0]][:4])


# (z, max_gapo, max_gape, seed_len, seed_z, end window)
LIMITS = [(0, 1, 2, 0, 0, 5), (1, 1, 0, 0, 0, 0), (2, 1, 2, 0, 0, 5), (2, 0, 3, 10, 1, 5), (3, 1, 6, 12, 1, 0),
          (3, 1, 2, 200, 2, 1), (4, 1, 6, 32, 2, 5), (5, 1, 3, 0, 0, 2), (6, 1, 2, 20, 0, 5), (1, 3, 6, 0, 0, 5)]


@pytest.mark.parametrize("name", ["iid", "repeats", "tandem", "short"])
@pytest.mark.parametrize("lim", LIMITS, ids=lambda x: "z%d_o%d_e%d_s%d_%d_w%d" % x)
def test_seed_search_equals_tree_search(torch, name, lim):
    z, go, ge, s, sz, e = lim
    text = _text(name)
    al = aln.Aligner(aln.Index.build(text, kmer_k=6).to_device(0))
    kw = dict(z=z, max_gapo=go, max_gape=ge, seed_len=s, seed_z=sz, indel_end_skip=e, mode=aln.MODE_PERSISTENT)
    sets = [((1, 2, 3, 5, 9, 14, 20, 31, 32, 33), 300), ((36, 50, 63, 64, 65, 76, 100), 500)]
    if z <= 4:
        sets.append(((128, 129, 150, 250, 255), 200))
    for i, (lengths, n) in enumerate(sets):
        lengths = tuple(x for x in lengths if x + 40 < text.size)
        reads = _reads(text, lengths, n, z, 50 + i)
        zz = (np.arange(reads.n) % (z + 1)).astype(np.uint8)
        for strata in (aln.STRATA_BEST1, aln.STRATA_FULL, aln.STRATA_SCORE):
            if strata != aln.STRATA_BEST1 and z > 3:
                continue
            for cap, zarr in ((255, None), (2, zz)):
                if min(lengths) < 9 and strata != aln.STRATA_BEST1 and z > 2:
                    continue  # every string of a few bases is within z: the tree search gives up on most
                p = aln.Params(hit_cap=cap, strata=strata, max_best=3 if cap == 2 else 0, **kw)
                got = al.align(reads.codes, reads.offsets, reads.lens, p, z=zarr)
                p.work_limit = TREE
                tree = al.align(reads.codes, reads.offsets, reads.lens, p, z=zarr)
                full = (tree[0]["flags"] & aln.FLAG_INCOMPLETE) != 0  # more candidates than the tree search keeps
                assert np.array_equal((got[0]["flags"] & aln.FLAG_INCOMPLETE) != 0, full), (name, lim, strata)
                keep = ~full
                _same((got[0][keep], got[1][keep]), (tree[0][keep], tree[1][keep]), cap, (name, lim, strata, i, cap))


@pytest.mark.parametrize("strata", [aln.STRATA_BEST1, aln.STRATA_FULL, aln.STRATA_SCORE])
def test_seed_search_against_the_oracle(torch, strata):
    """Repeats and tandems, one gap of up to three bases, the oracle's results."""
    for name in ("repeats", "tandem"):
        text = _text(name)
        ox = oracle.OracleIndex(text)
        al = aln.Aligner(aln.Index.build(text).to_device(0))
        lim = dict(z=3, max_gapo=1, max_gape=2, seed_len=20, seed_z=2, indel_end_skip=3)
        reads = _reads(text, (40, 64, 90), 400, 3, 9)
        kw = dict(score=(3, 11, 4), max_best=0) if strata == aln.STRATA_SCORE else {}
        ro, ho, _ = oracle_align(ox, reads, lim, 64, strata, **kw)
        p = aln.Params.from_limits(lim, hit_cap=64, strata=strata, mode=aln.MODE_PERSISTENT)
        rg, hg = al.align(reads.codes, reads.offsets, reads.lens, p)
        ok = (rg["flags"] & aln.FLAG_INCOMPLETE) == 0
        assert ok.mean() > 0.9
        compare(rg[ok], hg[ok], ro[ok], ho[ok], idx=np.nonzero(ok)[0], what=f"{name} {strata}")


def test_reads_left_to_the_tree_search(torch):
    """A text of one letter but for a random stretch: its reads have too many
    places for the seed search, in a batch with reads that have few: of up to
    2048 reads (the heavy phase in one kernel) and of more."""
    rng = Rng(5, "left")
    text = np.zeros(40_000, np.uint8)
    text[10_000:30_000] = reference_iid(20_000, rng.sub("t"))
    al = aln.Aligner(aln.Index.build(text, kmer_k=5).to_device(0))
    a = simulate_reads(text[10_000:30_000], 700, (50, 100), rng.sub("a"), z=2)
    b = Reads(np.zeros(64 * 40, np.uint8), np.arange(64, dtype=np.uint64) * np.uint64(40),
              np.full(64, 40, np.uint16), np.full(64, 2, np.uint8), np.zeros(64, np.int64), np.zeros(64, np.uint8))
    once = Reads.concat([a, b]).subset(np.random.default_rng(1).permutation(a.n + b.n))
    p = aln.Params(z=2, hit_cap=16, mode=aln.MODE_PERSISTENT)
    for reads in (once, Reads.concat([once] * 4)):
        for heavy in (0, 1, 0xFFFFFFFF):
            p.heavy_after, p.work_limit = heavy, 0
            got = al.align(reads.codes, reads.offsets, reads.lens, p)
            p.work_limit = TREE
            _same(got, al.align(reads.codes, reads.offsets, reads.lens, p), 16, heavy)
        assert (got[0]["c0"] > 9000).sum() >= 64
