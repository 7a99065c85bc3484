"""aln_pack_reads against packing base by base: lengths that leave words part
filled, empty reads (at the end too), scattered code offsets, codes above 4, and
batches large enough to be packed by several threads."""
import numpy as np
import pytest

import paper_1505_07855_gb300 as aln


def _reference(codes, offs, lens):
    at = np.repeat(offs.astype(np.int64) - (np.cumsum(lens, dtype=np.int64) - lens), lens)
    flat = codes[at + np.arange(at.size)]
    j = np.arange(flat.size)
    bases = np.zeros(max(1, (flat.size + 15) // 16), np.uint32)
    nmask = np.zeros(max(1, (flat.size + 31) // 32), np.uint32)
    np.bitwise_or.at(bases, j // 16, np.where(flat > 3, 0, flat).astype(np.uint32) << (2 * (j % 16)).astype(np.uint32))
    np.bitwise_or.at(nmask, j // 32, (flat > 3).astype(np.uint32) << (j % 32).astype(np.uint32))
    return bases, nmask


@pytest.mark.parametrize("n,most", [(0, 5), (1, 0), (1, 1), (3, 7), (50, 40), (1000, 255), (7000, 255)])
def test_pack_reads(n, most):
    rng = np.random.default_rng(n + most)
    for tail in (0, 3):
        lens = np.concatenate([rng.integers(0, most + 1, n), np.zeros(tail)]).astype(np.uint16)
        codes = rng.integers(0, 5, int(lens.sum()) + 300).astype(np.uint8)
        codes[rng.random(codes.size) < 0.02] = rng.integers(4, 256)
        offs = rng.integers(0, codes.size - 255, lens.size).astype(np.uint64)
        bases, nmask, at = aln.pack_reads(codes, offs, lens)
        rb, rn = _reference(codes, offs, lens)
        assert np.array_equal(bases, rb) and np.array_equal(nmask, rn)
        assert np.array_equal(at, (np.cumsum(lens, dtype=np.uint64) - lens))
