"""fm_index_load takes every image that fm_index_save wrote and refuses one whose
tables no longer agree with its symbols: device code follows an index's numbers
as rows, so a damaged file has to end at the loader (ALN_EIO).  No GPU."""
import numpy as np
import pytest

import paper_1505_07855_gb300 as aln
from synth import Rng, reference_iid

K, SAMPLE = 3, 4
HEAD, TEXT = 8 + 24, 48  # magic and (sa_sample, kmer_k, n_seed); (n, primary, C[4])


def _saved(tmp_path, n, sample=SAMPLE, kmer_k=K):
    path = str(tmp_path / "ix.bin")
    aln.Index.build(reference_iid(n, Rng(n, "file")), sa_sample=sample, kmer_k=kmer_k).save(path)
    return np.fromfile(path, np.uint8)


def _load(tmp_path, data):
    path = str(tmp_path / "q.bin")
    data.tofile(path)
    return aln.Index.load(path)


@pytest.mark.parametrize("n", [1, 2, 94, 95, 96, 97, 190, 191, 192, 193, 287, 288, 383, 384, 5000])
@pytest.mark.parametrize("kmer_k", [0, 4])
def test_saved_images_load(tmp_path, n, kmer_k):
    data = _saved(tmp_path, n, kmer_k=kmer_k)
    assert _load(tmp_path, data).info()["n"] == n


def test_large_image_loads(tmp_path):  # several ranges of samples and intervals
    assert _load(tmp_path, _saved(tmp_path, 400_000, sample=1, kmer_k=9)).info()["n"] == 400_000


def _vectors(data, text):
    """Byte offsets of a text's header and of its blocks, samples and intervals."""
    off = HEAD
    for t in range(text + 1):
        head, vec = off, []
        off += TEXT
        for _ in range(3):
            size = int(data[off:off + 8].view(np.uint64)[0])
            vec.append((off + 8, size))
            off += 8 + 4 * size
    return head, vec


@pytest.mark.parametrize("text", [0, 1])
@pytest.mark.parametrize("what", ["count", "count far", "plane", "plane of the last rows", "C", "C past the text", "primary",
                                  "primary elsewhere", "sample", "interval", "interval inverted", "sampling"])
def test_damaged_images_are_refused(tmp_path, what, text):
    n = 1000
    data = _saved(tmp_path, n).copy()
    head, ((blocks, n_words), (samp, n_samp), (kmer, n_kmer)) = _vectors(data, text)
    word = lambda off: data[off:off + 4].view(np.uint32)  # noqa: E731
    long = lambda off: data[off:off + 8].view(np.uint64)  # noqa: E731
    assert long(head)[0] == n and n_words == 16 * (1001 // 192 + 1)
    if what == "count":
        word(blocks + 64 * 2 + 4)[0] += 1
    elif what == "count far":
        word(blocks + 64 * 3)[0] = 0xFFFF0000
    elif what == "plane":
        word(blocks + 64 + 16)[0] ^= 1 << 9
    elif what == "plane of the last rows":  # rows 960..1000 lie in the last block
        word(blocks + 64 * 5 + 16)[0] ^= 1 << 3
    elif what == "C":
        long(head + 16 + 16)[0] += 1
    elif what == "C past the text":
        long(head + 16 + 24)[0] = 1 << 31
    elif what == "primary":
        long(head + 8)[0] = n + 1
    elif what == "primary elsewhere":  # at a row that holds another letter than A
        planes = data[blocks + 16:blocks + 16 + 24].view(np.uint32)
        rows = [r for r in range(96) if (planes[r // 32] | planes[3 + r // 32]) >> np.uint32(r % 32) & 1]
        long(head + 8)[0] = rows[0]
    elif what == "sample":
        word(samp + 4 * (n_samp // 2))[0] = n + 1
    elif what == "interval":
        word(kmer + 4 * (n_kmer // 2 + 1))[0] = n + 2
    elif what == "interval inverted":
        at = kmer + 8 * (n_kmer // 4)
        word(at)[0], word(at + 4)[0] = 7, 6
    elif what == "sampling":
        long(8)[0] = 3
    with pytest.raises(aln.AlnError) as e:
        _load(tmp_path, data)
    assert e.value.status == -6  # ALN_EIO
