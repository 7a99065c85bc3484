"""An index whose LF steps do not run through the whole text in one cycle (two of
its symbols swapped, its counts and samples made to fit, so that the loader has
nothing to refuse and every row it leads to exists): no walk from a sampled row
passes the rows of the other cycles, so nothing may be derived from it.  Their
positions end at the walk's bound, as they do from the image alone; the rows on
the sampled cycle keep theirs."""
import struct

import numpy as np
import pytest

import paper_1505_07855_gb300 as aln
from synth import Rng, reference_iid
from test_capi_host import _decode_bwt, _read_index_file

pytestmark = pytest.mark.gpu


def _lf(bwt, primary):
    """LF of every row, -1 at the row of $ (bwt has a 0 there)."""
    n = bwt.size - 1
    rows = np.arange(n + 1) != primary
    lf = np.full(n + 1, -1, np.int64)
    at = 1
    for c in range(4):
        of = np.nonzero(rows & (bwt == c))[0]
        lf[of] = at + np.arange(of.size)
        at += of.size
    return lf


def _steps_to_dollar(lf, primary):
    """LF steps from each row to the row of $, -1 where none lead there."""
    steps = np.full(lf.size, -1, np.int64)
    back = np.full(lf.size, -1, np.int64)
    back[lf[lf >= 0]] = np.nonzero(lf >= 0)[0]
    r, t = primary, 0
    while r >= 0:
        steps[r] = t
        r, t = back[r], t + 1
    return steps


def _blocks(bwt):
    """The image's Occ blocks: counts before the middle row, then bit planes."""
    nb = bwt.size // 192 + 1
    sym = np.zeros(nb * 192, np.uint32)
    sym[:bwt.size] = bwt
    out = np.zeros((nb, 16), np.uint32)
    for c in range(4):
        out[:, c] = np.concatenate([[0], np.cumsum(sym == c)])[np.arange(nb) * 192 + 96]
    bits = sym.reshape(nb, 2, 3, 32)
    for plane in (0, 1):
        w = (((bits >> plane) & 1) << np.arange(32, dtype=np.uint32)).sum(-1, dtype=np.uint64).astype(np.uint32)
        for half in (0, 1):
            out[:, 4 + 6 * half + 3 * plane:7 + 6 * half + 3 * plane] = w[:, half]
    return out


def test_nothing_is_derived_past_the_sampled_cycle(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n = 900
    path = str(tmp_path / "ix.bin")
    aln.Index.build(reference_iid(n, Rng(3, "cycle")), sa_sample=1024).save(path)
    f = _read_index_file(path)
    assert all(np.array_equal(_blocks(_decode_bwt(t)), t["blocks"]) for t in f["t"])
    bwt, primary = _decode_bwt(f["t"][0]), f["t"][0]["primary"]
    assert (_steps_to_dollar(_lf(bwt, primary), primary) >= 0).all()
    for j in range(400, n):
        b = bwt.copy()
        b[[300, j]] = b[[j, 300]]
        steps = _steps_to_dollar(_lf(b, primary), primary)
        if primary not in (300, j) and 200 < (steps < 0).sum() and steps[0] > 200:
            break
    f["t"][0].update(blocks=_blocks(b), sa=np.array([steps[0]], np.uint32))
    with open(path, "wb") as out:
        out.write(b"ALNFMIX4" + struct.pack("<3Q", f["sa_sample"], f["kmer_k"], f["n_seed"]))
        for t in f["t"]:
            out.write(struct.pack("<6Q", t["n"], t["primary"], *t["C"]))
            for v in (t["blocks"], t["sa"], t["kmer"]):
                out.write(struct.pack("<Q", v.size) + v.astype("<u4").tobytes())
    al = aln.Aligner(aln.Index.load(path).to_device(0))
    other = _decode_bwt(f["t"][1])
    exp = {1: steps, 0: _steps_to_dollar(_lf(other, f["t"][1]["primary"]), f["t"][1]["primary"])}
    for strand in (0, 1):
        hits = np.zeros(n + 1, aln.HIT_DTYPE)
        hits["k"] = hits["l"] = np.arange(n + 1)
        hits["strand"] = strand
        pos, npos = al.positions(hits, 1)
        lost = exp[strand] < 0
        assert (npos[lost] == aln.POS_WALK_LIMIT).all() and (npos[~lost] == 1).all()
        want = exp[strand] if strand else n - exp[strand]
        assert np.array_equal(pos[~lost, 0].astype(np.int64), want[~lost])
        assert lost.any() == bool(strand)
