"""Targets of several places that the seed search meets with more than one witness: a
gap beside a tandem may be placed on either side of a clean part, in families whose
copies meet in different rounds, and a target keeps its least witness before its
rows are joined to an interval (else a second, partial interval was reported; these
texts and reads are ones for which it was).  Against the oracle."""
import numpy as np
import pytest

import oracle
import paper_1505_07855_gb300 as aln
from parity_util import compare, oracle_align
from synth import Reads

pytestmark = pytest.mark.gpu


def _case(seed):
    g = np.random.default_rng(seed)
    text = g.integers(0, 4, 9000).astype(np.uint8)
    unit = g.integers(0, 4, g.integers(1, 4))
    fam = np.concatenate([g.integers(0, 4, 40), np.tile(unit, 12), g.integers(0, 4, 30), np.tile(g.integers(0, 4, 2), 8),
                          g.integers(0, 4, 40)]).astype(np.uint8)
    for i in range(int(g.integers(2, 30))):
        c = fam.copy()
        if i % 4 == 3:
            c[g.integers(0, c.size)] ^= 1
        text[200 + 260 * i:200 + 260 * i + c.size] = c
    g = np.random.default_rng(1000 + seed)
    reads = []
    for _ in range(60):  # pieces of the family with up to two edits
        m, a = int(g.integers(40, 110)), int(g.integers(0, fam.size - 30))
        c = fam[a:a + m].copy()
        for _ in range(int(g.integers(0, 3))):
            j, kind = int(g.integers(0, c.size)), g.integers(0, 3)
            if kind == 0:
                c[j] = (c[j] + 1) & 3
            elif kind == 1:
                c = np.delete(c, slice(j, j + int(g.integers(1, 3))))
            else:
                c = np.insert(c, j, g.integers(0, 4, g.integers(1, 3)))
        if g.random() < .5:
            c = 3 - c[::-1]
        if c.size >= 30:
            reads.append(Reads(c.astype(np.uint8), np.zeros(1, np.uint64), np.array([c.size], np.uint16),
                               np.array([3], np.uint8), np.zeros(1, np.int64), np.zeros(1, np.uint8)))
    return text, Reads.concat(reads), int(g.integers(0, 6))


@pytest.mark.parametrize("seed", [1, 20, 27, 36, 38])
@pytest.mark.parametrize("strata", [aln.STRATA_BEST1, aln.STRATA_FULL])
def test_one_interval_a_target(seed, strata):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    text, reads, e = _case(seed)
    lim = dict(z=3, max_gapo=1, max_gape=2, seed_len=0, seed_z=0, indel_end_skip=e)
    ro, ho, _ = oracle_align(oracle.OracleIndex(text), reads, lim, 64, strata)
    al = aln.Aligner(aln.Index.build(text).to_device(0))
    for mode in (aln.MODE_PERSISTENT, aln.MODE_PLAIN):
        p = aln.Params.from_limits(lim, hit_cap=64, strata=strata, mode=mode)
        compare(*al.align(reads.codes, reads.offsets, reads.lens, p), ro, ho, what=f"{seed} {strata} {mode}")
