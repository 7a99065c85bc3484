"""Reads that the heavy phase searches in earnest: each has a hundred and more
distinct hits (variants of one sequence, more than a block's threads), listed in
full, cut at the hit cap, and counted; every field against the oracle.  The reads
reach it in both of its forms: one kernel a pass, in a call whose reads all go to
the tree search (a work limit is set), and the whole phase in one kernel, in a call
of at most 2048 reads that the seed search leaves (17 000 places each).  The
number handed over is read from the call's own scratch."""
import numpy as np
import pytest

import oracle
import paper_1505_07855_gb300 as aln
from parity_util import compare, oracle_align
from synth import Reads, Rng, reference_iid

pytestmark = pytest.mark.gpu
COPIES, LEN, VARIANTS = 17_000, 48, 150


@pytest.fixture(scope="module")
def family():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    g = np.random.default_rng(12)
    rng = Rng(12, "variants")
    unit = reference_iid(LEN, rng.sub("u"))
    # VARIANTS - 1 single substitutions over the whole unit, and the unit itself
    at = np.arange(1, VARIANTS) % LEN
    kinds = np.repeat(unit[None], VARIANTS, 0)
    kinds[np.arange(1, VARIANTS), at] = (unit[at] + 1 + np.arange(1, VARIANTS) // LEN) & 3
    text = reference_iid(COPIES * (LEN + 9), rng.sub("t")).reshape(COPIES, LEN + 9)
    text[:, :LEN] = kinds[g.integers(0, VARIANTS, COPIES)]
    text = np.ascontiguousarray(text.reshape(-1))
    n = 300
    codes = np.repeat(unit[None], n, 0)
    codes[100:200] = kinds[g.integers(0, VARIANTS, 100)]
    codes[::2] = 3 - codes[::2, ::-1]
    reads = Reads(codes.reshape(-1), np.arange(n, dtype=np.uint64) * np.uint64(LEN), np.full(n, LEN, np.uint16),
                  np.full(n, 2, np.uint8), np.zeros(n, np.int64), np.zeros(n, np.uint8))
    return torch, oracle.OracleIndex(text), aln.Aligner(aln.Index.build(text, kmer_k=6).to_device(0)), reads


@pytest.mark.parametrize("cap", [1, 7, 255])
@pytest.mark.parametrize("strata,max_best", [(aln.STRATA_BEST1, 0), (aln.STRATA_FULL, 0), (aln.STRATA_SCORE, 0),
                                             (aln.STRATA_SCORE, 20)])
def test_heavy_reads_with_many_hits(family, strata, max_best, cap):
    torch, ox, al, reads = family
    lim = dict(z=2 if strata == aln.STRATA_BEST1 else 1, max_gapo=0, max_gape=0, seed_len=0, seed_z=0, indel_end_skip=5)
    kw = dict(score=(3, 11, 4), max_best=max_best) if strata == aln.STRATA_SCORE else {}
    ro, ho, _ = oracle_align(ox, reads, lim, cap, strata, **kw)
    n = reads.n
    d = al.upload(reads.codes, reads.offsets, reads.lens)
    res, hits = al.outputs(n, cap)
    for work_limit in (1 << 24, 0):
        p = aln.Params.from_limits(lim, hit_cap=cap, strata=strata, mode=aln.MODE_PERSISTENT, heavy_after=1,
                                   work_limit=work_limit, max_best=max_best)
        scratch = torch.zeros(aln.scratch_bytes(n), dtype=torch.uint8, device="cuda")
        al.search_device(d, p, res, hits, scratch=scratch)
        r = res.cpu().numpy().view(aln.RES_DTYPE)[:n]
        h = hits.cpu().numpy().view(aln.HIT_DTYPE)[:n * cap].reshape(n, cap)
        compare(r, h, ro, ho, what=f"{strata} {cap} {work_limit}")
        header = (256 + 20 * n + 255) // 256 * 256  # the heavy phase's state lies behind the order
        assert int(scratch[header:header + 4].cpu().numpy().view(np.uint32)[0]) > n // 2
    if cap == 255 and not max_best:
        assert (r["n_hits"] > 128).sum() >= 200
