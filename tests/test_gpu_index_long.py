"""A text long enough for the GPU builder's 24-symbol first round (2^29 bases and
more): every row of both suffix arrays, located through the uploaded index, is
checked by the definition: the rows are a permutation of the positions, and each
suffix is below the next one (by its first base, or where those are equal by the
rows of the suffixes one base shorter).  The rows between the samples come from
LF steps, so the Occ blocks are checked with them."""
import numpy as np
import pytest

import paper_1505_07855_gb300 as aln

pytestmark = pytest.mark.gpu


def test_every_row_of_a_long_text():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n = (1 << 29) + 77
    g = np.random.default_rng(29)
    text = g.integers(0, 4, n, dtype=np.uint8)
    unit = text[:5000].copy()
    for at in g.integers(10_000, n - 10_000, 300):  # copies, tandems and one long run: the doubling rounds
        text[at:at + 5000] = unit
    text[1 << 28:(1 << 28) + 6000] = np.tile(unit[:3], 2000)
    text[(1 << 28) + 9000:(1 << 28) + 11_000] = 0
    text[-40:] = text[100:140]
    al = aln.Aligner(aln.Index.build(text, device=0).to_device(0))
    assert al.dix.derived_bytes() > 14 * n
    x = torch.from_numpy(text).cuda()
    for strand in (1, 0):  # the suffix arrays of the text and of the text reversed
        y = x if strand else x.flip(0)
        sa = torch.empty(n + 1, dtype=torch.int64, device="cuda")
        for a in range(0, n + 1, 1 << 26):
            rows = torch.arange(a, min(a + (1 << 26), n + 1), device="cuda", dtype=torch.int32)
            hits = torch.zeros(rows.numel(), 4, dtype=torch.int32, device="cuda")
            hits[:, 0] = hits[:, 1] = rows
            hits[:, 2] = strand << 16
            npos = torch.empty(rows.numel(), dtype=torch.int32, device="cuda")
            al.dix.sa_to_pos(hits, rows.numel(), 1, sa[a:a + rows.numel()], npos)
            assert (npos == 1).all()
        if not strand:
            sa = n - sa
        assert int(sa[0]) == n
        row = torch.full((n + 1,), -1, dtype=torch.int32, device="cuda")
        row[sa] = torch.arange(n + 1, device="cuda", dtype=torch.int32)
        assert (row >= 0).all()
        i, j = sa[1:-1], sa[2:]  # row 0 is "$"
        first, then = y[i], y[j]
        assert (first <= then).all()
        same = first == then
        assert (row[i[same] + 1] < row[j[same] + 1]).all()
        del sa, row, i, j, first, then, same
