"""The tree search at work on every read of a batch: with the default work limit given
explicitly no read is answered from seeds, so the schedule's knobs, the shared
stacks, the heavy phase, the visit order and the server search the batches they
were written for (without the limit most of their reads never reach them).  Results
against the oracle; where the heavy phase is the subject, the number of reads
handed over is read from the call's scratch.  And the other way round: the seed
search at the largest budget, 7 differences over 8 parts."""
import numpy as np
import pytest

import oracle
import paper_1505_07855_gb300 as aln
from parity_util import compare, oracle_align
from synth import Rng, reference_iid, simulate_reads, workload
from test_gpu_parity import LIMITS, Pair
from test_gpu_seed import TREE, _reads, _same, _text
from test_gpu_serving import _requests
from test_gpu_serving import _same as same_hits

pytestmark = pytest.mark.gpu
M = [20, 36, 50, 36, 60, 76, 40]  # read lengths of LIMITS


@pytest.fixture(scope="module")
def cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


def _search(torch, al, reads, p, z=None):
    """Results, and the reads handed over to the heavy phase."""
    d = al.upload(reads.codes, reads.offsets, reads.lens, z)
    res, hits = al.outputs(d["n"], p.hit_cap)
    scratch = torch.zeros(aln.scratch_bytes(d["n"]), dtype=torch.uint8, device="cuda")
    al.search_device(d, p, res, hits, scratch=scratch)
    al.check_status()
    n = d["n"]
    header = (256 + 20 * n + 255) // 256 * 256
    return (res.cpu().numpy().view(aln.RES_DTYPE)[:n],
            hits.cpu().numpy().view(aln.HIT_DTYPE)[:n * p.hit_cap].reshape(n, p.hit_cap),
            int(scratch[header:header + 4].cpu().numpy().view(np.uint32)[0]))


@pytest.fixture(scope="module")
def mixed(cuda):
    w = workload("human_mixed", ref_len=3_000_000, n_reads=3000, seed=3)
    pair = Pair(w.text, n_seed=7, kmers=[11])
    return w, pair, oracle_align(pair.ox, w.reads, w.params, 32, oracle.BEST1, z=w.reads.z)[:2]


@pytest.mark.parametrize("help_after,smem,bps,win,heavy", [
    (0, 0, 0, 0, 0), (1, 4, 0, 0, 0), (0xFFFFFFFF, 12, 0, 1, 1), (64, 8, 1, 0, 64), (0, 12, 2, 1, 0xFFFFFFFF)])
def test_schedule_knobs(cuda, mixed, help_after, smem, bps, win, heavy):
    w, pair, (ro, ho) = mixed
    p = aln.Params.from_limits(w.params, hit_cap=32, mode=aln.MODE_PERSISTENT, z=6, help_after=help_after, smem_stack=smem,
                               blocks_per_sm=bps, l2_window=win, heavy_after=heavy, work_limit=TREE)
    rg, hg, handed = _search(cuda, pair.al, w.reads, p, w.reads.z)
    compare(rg, hg, ro, ho, what="mixed")
    if heavy == 1:
        assert handed > 500


@pytest.mark.parametrize("mode", [aln.MODE_PLAIN, aln.MODE_PERSISTENT])
def test_read_order(cuda, mixed, mode):
    w, pair, (ro, ho) = mixed
    perm = np.random.default_rng(4).permutation(w.reads.n)
    sub = w.reads.subset(perm)
    p = aln.Params.from_limits(w.params, hit_cap=32, mode=mode, z=6, work_limit=TREE)
    rg, hg = pair.al.align(sub.codes, sub.offsets, sub.lens, p, z=sub.z)
    compare(rg, hg, ro[perm], ho[perm], idx=perm, what="permuted")


@pytest.mark.parametrize("li", [1, 4])
@pytest.mark.parametrize("strata", [aln.STRATA_BEST1, aln.STRATA_FULL, aln.STRATA_SCORE])
def test_heavy_phase(cuda, li, strata):
    lim = LIMITS[li]
    rng = Rng(5000 + li, "heavy")
    text = reference_iid(30_000, rng.sub("t"))
    text[9000:9400] = text[5000:5400] = text[1000:1400]  # repeats, so that best places tie
    pair = Pair(text, kmers=[0, 6])
    reads = simulate_reads(text, 2500, M[li], rng.sub("r"), sub_rate=(0.02, 0.04), indel_rate=0.005, indel_lens=(1, 2),
                           n_frac=0.1, z=lim["z"])
    kw = dict(score=(3, 11, 4), max_best=2) if strata == aln.STRATA_SCORE else {}
    ro, ho, _ = oracle_align(pair.ox, reads, lim, 40, strata, **kw)
    for k, heavy in ((0, 1), (6, 1), (6, 0)):
        p = aln.Params.from_limits(lim, hit_cap=40, strata=strata, mode=aln.MODE_PERSISTENT, heavy_after=heavy,
                                   max_best=kw.get("max_best", 0), work_limit=TREE)
        rg, hg, handed = _search(cuda, pair.als[k], reads, p)
        compare(rg, hg, ro, ho, what=f"limits {li} kmer {k} heavy_after {heavy}")
        assert handed > 1000 if heavy else handed == 0
    assert not kw or (rg["flags"] & aln.FLAG_MANY_BEST).any()


@pytest.mark.parametrize("heavy", [0, 1])
def test_server(cuda, mixed, heavy):
    w, pair, _ = mixed
    p = aln.Params.from_limits(w.params, hit_cap=8, mode=aln.MODE_PERSISTENT, z=6, heavy_after=heavy, work_limit=TREE)
    reqs = _requests(w, 12, 3)
    srv = aln.Server(pair.al.dix, p, n_slots=3, max_batch_reads=1500, coalesce_us=100)
    try:
        ids = [srv.submit(r.codes, r.offsets, r.lens, r.z) for r in reqs]
        got = [srv.poll(i, r.n)[:2] for i, r in zip(ids, reqs)]
    finally:
        srv.close()
    for r, g in zip(reqs, got):
        same_hits(pair.al.align(r.codes, r.offsets, r.lens, p, z=r.z), g, 8)


@pytest.mark.parametrize("mode", [aln.MODE_PLAIN, aln.MODE_PERSISTENT])
def test_seed_search_of_seven_differences(cuda, mode):
    """z = 7, one gap: the eight parts of 16 lanes; reads of up to seven errors."""
    text = _text("iid")[:30_000]
    al = aln.Aligner(aln.Index.build(text, kmer_k=6).to_device(0))
    g = np.random.default_rng(7)
    reads = _reads(text, (100,), 150, 7, 70)
    for i in range(reads.n):  # up to five more substitutions a read
        o, m = int(reads.offsets[i]), int(reads.lens[i])
        at = g.integers(0, m, i % 6)
        reads.codes[o + at] = g.integers(0, 4, at.size)
    p = aln.Params(z=7, max_gapo=1, max_gape=3, indel_end_skip=3, hit_cap=64, mode=mode)
    zz = (1 + np.arange(reads.n) % 7).astype(np.uint8)
    for z in (None, zz):
        got = al.align(reads.codes, reads.offsets, reads.lens, p, z=z)
        p.work_limit = TREE
        tree = al.align(reads.codes, reads.offsets, reads.lens, p, z=z)
        p.work_limit = 0
        assert not (tree[0]["flags"] & aln.FLAG_INCOMPLETE).any()
        _same(got, tree, 64, "z = 7")
    d = got[0]["d_best"]
    assert ((d >= 4) & (d < 255)).sum() > 20
