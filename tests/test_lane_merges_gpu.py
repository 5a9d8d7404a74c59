"""Merges a thread per piece: every length, at the numbers of pieces where k_merge and k_merge_bulk turn to it, against the oracle."""
import numpy as np
import pytest

from gpu_util import cpu_vocab, gpu_encode, gpu_vocab, same

pytestmark = pytest.mark.gpu


def _words(rng, lengths, alphabet):
    """Words of the given lengths with a line feed behind each (no word takes it in)."""
    letters = rng.choice(np.frombuffer(alphabet, dtype=np.uint8), int(lengths.sum()) + lengths.size)
    letters[np.cumsum(lengths + 1) - 1] = 10
    return letters


def _warps():
    import torch
    return 24 * torch.cuda.get_device_properties(0).multi_processor_count


# few letters: many equal ranks and tokens of many bytes, so that the order of equal pairs and every neighbour matters
@pytest.mark.parametrize("name", ["C1", "C4"])
@pytest.mark.parametrize("alphabet", [b"a", b"es", b"etaoinshr"])
@pytest.mark.parametrize("lo,hi,per_warp", [(2, 32, 1.9), (2, 32, 2.2), (2, 10, 5), (15, 18, 3), (31, 34, 9), (33, 64, 3.9), (33, 64, 4.2), (47, 49, 6), (60, 70, 9), (2, 80, 12)])
def test_words_of_every_length(name, alphabet, lo, hi, per_warp):
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
