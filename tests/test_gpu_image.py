"""An index uploaded without the arrays derived from it: every call gives the results
it gives with them, and both uploads tell what they hold.  A text whose LF walks
are too long to derive from (200 bases, 64 times: consecutive positions lie in
different groups of the suffix array, and all groups are aligned to the sampling)
is served the same way, the walks of its positions ending at their bound."""
import ctypes

import numpy as np
import pytest

import oracle
import paper_1505_07855_gb300 as aln
from parity_util import compare, oracle_align
from synth import Rng, reference_iid, simulate_reads, workload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    return t


@pytest.mark.parametrize("strata", [aln.STRATA_BEST1, aln.STRATA_FULL, aln.STRATA_SCORE])
def test_searches_and_positions_of_the_image_alone(torch, strata):
    w = workload("tiny36", ref_len=150_000, n_reads=2500, seed=8)
    idx = aln.Index.build(w.text, kmer_k=6)
    with_, alone = aln.Aligner(idx.to_device(0)), aln.Aligner(idx.to_device(0, derived=False))
    n = w.text.size
    assert alone.dix.derived_bytes() == 0 and alone.dix.info() == with_.dix.info()
    assert 14 * n < with_.dix.derived_bytes() < 30 * n
    assert aln.lib().fm_dindex_derived_bytes(None) == 0
    out = ctypes.c_void_p()
    assert aln.lib().fm_index_to_device_image(None, 0, None, ctypes.byref(out)) == -1
    kw = dict(score=(3, 11, 4), max_best=0) if strata == aln.STRATA_SCORE else {}
    ro, ho, _ = oracle_align(oracle.OracleIndex(w.text), w.reads, w.params, 8, strata, **kw)
    for mode in ([aln.MODE_PERSISTENT] if kw else [aln.MODE_PLAIN, aln.MODE_PERSISTENT]):
        for al in (alone, with_):
            p = aln.Params.from_limits(w.params, hit_cap=8, strata=strata, mode=mode)
            r, h = al.align(w.reads.codes, w.reads.offsets, w.reads.lens, p)
            compare(r, h, ro, ho, what=f"{strata} {mode}")
    hits = h[np.arange(8)[None, :] < r["n_hits"][:, None]]
    (pa, na), (pb, nb) = alone.positions(hits, 16), with_.positions(hits, 16)
    assert np.array_equal(na, nb)
    ok = np.arange(16)[None, :] < np.where(na <= 16, na, 0)[:, None]
    assert ok.any() and np.array_equal(pa[ok], pb[ok])


def _longest_walk(sa, sample):
    """Most LF steps from a row to one whose number the sampling keeps."""
    row = np.empty(sa.size, np.int64)
    row[sa] = np.arange(sa.size)
    kept = np.nonzero(row % sample == 0)[0]  # text positions in order; LF goes down
    return int(max(np.diff(kept).max(), sa.size - kept[-1]))


def test_text_too_long_to_walk(torch):
    text = np.tile(reference_iid(200, Rng(5, "period")), 64)
    ox = oracle.OracleIndex(text)
    assert _longest_walk(ox.sa(0), 32) > 64 * 32
    al = aln.Aligner(aln.Index.build(text, kmer_k=4).to_device(0))
    assert al.dix.derived_bytes() == 0
    reads = simulate_reads(text, 500, (36, 80), Rng(6, "reads"), sub_rate=(0.01, 0.03), indel_rate=0.005, z=2)
    lim = dict(z=2, max_gapo=1, max_gape=2, seed_len=0, seed_z=0, indel_end_skip=5)
    ro, ho, _ = oracle_align(ox, reads, lim, 16, oracle.BEST1)
    for mode in (aln.MODE_PLAIN, aln.MODE_PERSISTENT):
        r, h = al.align(reads.codes, reads.offsets, reads.lens, aln.Params.from_limits(lim, hit_cap=16, mode=mode))
        compare(r, h, ro, ho, what=f"period, mode {mode}")
    n = text.size
    hits = np.zeros(n + 1, aln.HIT_DTYPE)
    hits["k"] = hits["l"] = np.arange(n + 1)
    for strand, sa in ((1, ox.sa(0)), (0, ox.sa(1))):
        hits["strand"] = strand
        pos, npos = al.positions(hits, 1)
        ok = npos == 1
        assert ok.any() and (npos[~ok] == aln.POS_WALK_LIMIT).all()
        assert np.array_equal(pos[ok, 0].astype(np.int64), (sa if strand else n - sa.astype(np.int64))[ok])


def test_period_of_two_is_derived(torch):
    """Its walks stay far below the bound, so every row has a position."""
    text = np.tile(np.array([0, 3], np.uint8), 20_000)
    ox = oracle.OracleIndex(text)
    assert _longest_walk(ox.sa(0), 32) < 64 * 32
    al = aln.Aligner(aln.Index.build(text).to_device(0))
    assert al.dix.derived_bytes() > 0
    n = text.size
    hits = np.zeros(n + 1, aln.HIT_DTYPE)
    hits["k"] = hits["l"] = np.arange(n + 1)
    for strand, sa in ((1, ox.sa(0)), (0, ox.sa(1))):
        hits["strand"] = strand
        pos, npos = al.positions(hits, 1)
        assert (npos == 1).all()
        assert np.array_equal(pos[:, 0].astype(np.int64), sa.astype(np.int64) if strand else n - sa.astype(np.int64))
