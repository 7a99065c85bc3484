"""The autotuner's cache: a call returns what was measured for its own search.  A
loop or work limit selects the tree search, heavy_after, help_after and l2_window
how it runs, so a call that differs in one of them is timed anew (the searches it
times write the sample's results), and a repeated one is not."""
import pytest

import paper_1505_07855_gb300 as aln
from synth import workload

pytestmark = pytest.mark.gpu


def test_each_search_has_its_own_entry():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    w = workload("tiny36", ref_len=200_000, n_reads=3000, seed=5)
    al = aln.Aligner(aln.Index.build(w.text, kmer_k=6).to_device(0))
    d = al.upload(w.reads.codes, w.reads.offsets, w.reads.lens)
    res, hits = al.outputs(d["n"], 8)
    ms = {}
    for name, kw in (("loop limit", dict(loop_limit=1 << 30)), ("default", {}), ("work limit", dict(work_limit=1 << 24)),
                     ("no heavy phase", dict(heavy_after=0xFFFFFFFF)), ("help", dict(help_after=64)),
                     ("window", dict(l2_window=1))):
        p = aln.Params.from_limits(w.params, hit_cap=8, mode=aln.MODE_PERSISTENT, **kw)
        res.fill_(0xEE)
        tuned, ms[name] = al.autotune(d, p, res, hits)
        assert not (res == 0xEE).all(), f"{name}: another search's entry"
        res.fill_(0xEE)
        assert al.autotune(d, p, res, hits) == (tuned, ms[name]) and (res == 0xEE).all()
    assert ms["loop limit"] > 2 * ms["default"]  # the tree search of every read, and the seed search
