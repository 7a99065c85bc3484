"""sa_to_pos from the whole suffix array (derived on the device at upload) and
from the walk over the sampled one give the same numbers: both against the
oracle's suffix arrays, over every row of texts whose walks are short, long, or
too long for the derivation (a two-letter period: its rows jump between the two
halves of the array)."""
import numpy as np
import pytest

import oracle
import paper_1505_07855_gb300 as aln
from synth import Rng, reference_iid

pytestmark = pytest.mark.gpu


def _texts():
    rng = Rng(77, "derived")
    yield "one base", np.array([2], np.uint8), 32
    yield "ragged", reference_iid(1000 + 193, rng.sub("a")), 32
    yield "every row sampled", reference_iid(777, rng.sub("b")), 1
    yield "few rows sampled", reference_iid(40_000, rng.sub("c")), 1024
    yield "one letter", np.zeros(5000, np.uint8), 32
    yield "period 2", np.tile(np.array([0, 3], np.uint8), 20_000), 32


@pytest.mark.parametrize("width", [1, 2, 33, 64])
def test_positions_of_every_row(width):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    for name, text, sample in _texts():
        n = text.size
        ox = oracle.OracleIndex(text)
        al = aln.Aligner(aln.Index.build(text, sa_sample=sample).to_device(0))
        k = np.arange(0, n + 1, max(1, (n + 1) // 700), dtype=np.int64)
        w = np.minimum(1 + k % (width + 1), n + 1 - k)  # widths 1 .. width + 1: the last is too wide
        hits = np.zeros(2 * k.size, aln.HIT_DTYPE)
        oh = np.zeros(hits.size, oracle.HIT_DTYPE)
        for h in (hits, oh):
            h["k"] = np.concatenate([k, k])
            h["l"] = np.concatenate([k + w - 1, k + w - 1])
            h["strand"] = np.repeat([0, 1], k.size)
            h["aligned_len"] = 0
        opos, onpos = ox.positions(oh, width)
        for shift in (0, 4):  # 16-byte records, and records off that boundary (the walk)
            raw = torch.zeros(shift + hits.nbytes, dtype=torch.uint8, device="cuda")
            raw[shift:] = torch.from_numpy(hits.view(np.uint8)).cuda()
            pos = torch.zeros(hits.size * width, dtype=torch.int64, device="cuda")
            npos = torch.zeros(hits.size, dtype=torch.int32, device="cuda")
            al.dix.sa_to_pos(raw[shift:], hits.size, width, pos, npos)
            gp = pos.cpu().numpy().view(np.uint64).reshape(hits.size, width)
            gn = npos.cpu().numpy().view(np.uint32)
            wide = np.concatenate([w, w]) > width
            assert (gn[wide] == aln.POS_TOO_WIDE).all(), name
            ok = ~wide & (gn != aln.POS_WALK_LIMIT)
            assert name == "period 2" or ok[~wide].all(), name
            assert np.array_equal(gn[ok], onpos[ok]), name
            for i in np.nonzero(ok)[0]:
                assert np.array_equal(gp[i, :gn[i]], opos[i, :gn[i]]), (name, shift, i)
