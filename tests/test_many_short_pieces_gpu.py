"""More short pieces than the rule of k_merge gives to warps: batches of them, a thread each."""
import numpy as np
import pytest

import workloads as wl
from gpu_util import at_the_merge_rule, cpu_vocab, gpu_encode, gpu_vocab, same, to_dev

pytestmark = pytest.mark.gpu


def _words(rng, k, n):
    w = (97 + rng.integers(0, 26, (n, k + 1))).astype(np.uint8)
    w[:, k] = 32
    return w.ravel()


# just below the rule, just above it, and with many times as many pieces
@pytest.mark.parametrize("name", ["C1", "C4"])
@pytest.mark.parametrize("size,n", [(4, 0), (9, 0), (20, 0), (30, 0), (4, 43_000), (9, 42_300), (2, 130_000), (20, 43_001), (30, 44_000)])
def test_words_around_the_limit(name, size, n):
    rng = np.random.default_rng(size * 1000 + n)
    gv, cv = gpu_vocab(name), cpu_vocab(name)
    offset = n % 16
    texts = [_words(rng, size, n)[: n * (size + 1) - 1]] if n else at_the_merge_rule(cv, _words(rng, size, 120_000 // (size // 10 + 1)), gv.pattern_id, offset)
    for text in texts:
        ids, status = gpu_encode(gv, text, offset=offset)
        assert status == 0 and same(ids, cv.encode(text, gv.pattern_id, nthreads=8)[0])


@pytest.mark.parametrize("name", ["C1", "C4"])
def test_with_long_pieces_among_them(name):
    """Then the batches go by tickets: long pieces of a CTA's size and of the whole grid's."""
    rng = np.random.default_rng(7)
    gv, cv = gpu_vocab(name), cpu_vocab(name)
    for long in (300, 4_000, 70_000):
        text = np.r_[_words(rng, 5, 30_000), (97 + rng.integers(0, 26, long)).astype(np.uint8), np.uint8([10]), _words(rng, 7, 30_000)]
        ids, status = gpu_encode(gv, text)
        assert status == 0 and same(ids, cv.encode(text, gv.pattern_id, nthreads=8)[0]), long


def test_two_byte_pieces_use_the_whole_gpu():
    import torch
    gv, cv = gpu_vocab("C4"), cpu_vocab("C4")
    text = np.frombuffer(b" ." * 150_000, dtype=np.uint8)
    d, bufs = to_dev(text), gv.alloc(text.size)
    ms = np.median([gv.encode_timed(d, bufs)["merge"] for _ in range(11)])
    torch.cuda.synchronize()
    assert same(bufs["ids"][:int(bufs["count"])].cpu().numpy(), cv.encode(text, 1)[0])
    # 0.065 ms; 0.118 to 0.137 where a warp took the pieces of a whole tile
    assert ms < 0.095, ms
