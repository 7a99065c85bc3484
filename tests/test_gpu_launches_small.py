"""The kernels of one persistent search, counted by the CUDA profiler, against
bench.search_launches for a call's number of reads: up to 2048 the heavy phase of a
seed search is one kernel, past that and in a call whose reads all go to the tree
search it is eleven."""
import pytest

import paper_1505_07855_gb300 as aln
from synth import workload
from test_gpu_launches import _kernels

pytestmark = pytest.mark.gpu


def test_launches_follow_the_number_of_reads():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import bench
    w = workload("tiny36", ref_len=100_000, n_reads=2049, seed=22)
    al = aln.Aligner(aln.Index.build(w.text).to_device(0))
    seen = set()
    for n in (1, 2048, 2049):
        r = w.reads.subset(range(n))
        d = al.upload(r.codes, r.offsets, r.lens)
        res, hits = al.outputs(n, 8)
        for kw in ({}, dict(work_limit=1 << 24), dict(loop_limit=1 << 30), dict(max_gapo=2), dict(heavy_after=0xFFFFFFFF)):
            p = aln.Params.from_limits(w.params, **dict(dict(hit_cap=8, mode=aln.MODE_PERSISTENT), **kw))
            for _ in range(2):  # warm-up; the profiler's first session can miss kernels
                got = _kernels(torch, lambda: al.search_device(d, p, res, hits))
            assert len(got) == bench.search_launches(aln, p, n_reads=n), (n, kw, got)
            seen.add(len(got))
    assert seen == {4, 5, 4 + 1 + 2 * aln.HEAVY_PASSES}
