"""Merges a thread per piece: every length, on either side of the rule by which k_merge turns to them, and in bulk text, against the oracle."""
import numpy as np
import pytest

from gpu_util import at_the_merge_rule, cpu_vocab, gpu_encode, gpu_vocab, same

pytestmark = pytest.mark.gpu


def _words(rng, lengths, alphabet):
    """Words of the given lengths with a line feed behind each (no word takes it in)."""
    letters = rng.choice(np.frombuffer(alphabet, dtype=np.uint8), int(lengths.sum()) + lengths.size)
    letters[np.cumsum(lengths + 1) - 1] = 10
    return letters


def _warps():
    import torch
    return 24 * torch.cuda.get_device_properties(0).multi_processor_count


# few letters: many equal ranks and tokens of many bytes, so that the order of equal pairs and every neighbour matters; the last text that goes a warp
# per piece and the first one that goes a thread per piece, with pieces of up to 16 bytes (half the columns), around 16 and up to 32
@pytest.mark.parametrize("name", ["C1", "C4"])
@pytest.mark.parametrize("alphabet", [b"es", b"qxz", b"etaoinshr"])
@pytest.mark.parametrize("lo,hi", [(2, 32), (2, 10), (8, 16), (15, 18), (17, 24), (31, 32)])
def test_words_of_every_length(name, alphabet, lo, hi):
    rng = np.random.default_rng(lo * 100 + hi)
    gv, cv = gpu_vocab(name), cpu_vocab(name)
    offset = (lo + hi) % 16
    text = _words(rng, rng.integers(lo, hi + 1, 15 * _warps()), alphabet)
    for cut in at_the_merge_rule(cv, text[:4_000_000], gv.pattern_id, offset):
        ids, status = gpu_encode(gv, cut, offset=offset)
        assert status == 0 and same(ids, cv.encode(cut, gv.pattern_id, nthreads=8)[0])


# the same word over and over: all threads of a batch in step
@pytest.mark.parametrize("name", ["C1", "C4"])
@pytest.mark.parametrize("size", [25, 31, 32])
def test_one_letter_words(name, size):
    gv, cv = gpu_vocab(name), cpu_vocab(name)
    text = _words(np.random.default_rng(size), np.full(8 * _warps(), size), b"a")
    ids, status = gpu_encode(gv, text)
    assert status == 0 and same(ids, cv.encode(text, gv.pattern_id, nthreads=8)[0])


# among longer pieces, a warp each: short and long ones in one text, and only long ones
@pytest.mark.parametrize("name", ["C1", "C4"])
@pytest.mark.parametrize("alphabet", [b"a", b"es", b"etaoinshr"])
@pytest.mark.parametrize("lo,hi,per_warp", [(31, 34, 9), (33, 64, 3.9), (33, 64, 4.2), (47, 49, 6), (60, 70, 9), (2, 80, 12)])
def test_words_of_more_than_32_bytes(name, alphabet, lo, hi, per_warp):
    rng = np.random.default_rng(lo * 100 + hi)
    gv, cv = gpu_vocab(name), cpu_vocab(name)
    text = _words(rng, rng.integers(lo, hi + 1, int(per_warp * _warps())), alphabet)
    ids, status = gpu_encode(gv, text, offset=(lo + hi) % 16)
    assert status == 0 and same(ids, cv.encode(text, gv.pattern_id, nthreads=8)[0])


# more than 4 MB: the lists of bulk text, with few and with many pieces of a class
@pytest.mark.parametrize("name", ["C1", "C4"])
@pytest.mark.parametrize("lo,hi,size", [(2, 32, 5_000_000), (30, 66, 5_000_000), (33, 64, 6_000_000), (100, 250, 5_000_000)])
def test_bulk_words_of_every_length(name, lo, hi, size):
    rng = np.random.default_rng(lo + hi)
    gv, cv = gpu_vocab(name), cpu_vocab(name)
    text = _words(rng, rng.integers(lo, hi + 1, 2 * size // (lo + hi)), b"etaoinshr")
    ids, status = gpu_encode(gv, text)
    assert status == 0 and same(ids, cv.encode(text, gv.pattern_id, nthreads=8)[0])
