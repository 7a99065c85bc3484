"""Where the persistent form's seed search sends a read, from the counts at the start
of the call's scratch (reads left for more lanes, taken up there, left for the
tree): few places are answered at once, hundreds by a warp, a read with more targets than a
warp keeps goes on to the tree search, and one with more places than a warp looks at
goes there without that try."""
import numpy as np
import pytest

import paper_1505_07855_gb300 as aln
from synth import Rng, reference_iid

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
