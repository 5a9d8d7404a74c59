"""GPU merges of pieces of more than 256 bytes against the oracle, exact: windows of 256 bytes every 192 that are joined at
shared tokens, pieces of at most 32 byte runs merged as runs, and what neither settles (windows that do not meet)."""
import numpy as np
import pytest

from gpu_util import cpu_vocab, gpu_encode, gpu_encode_batch, gpu_vocab, same

pytestmark = pytest.mark.gpu

# one window and one byte more, the second and third window's edges (256 + 192 k, and 64 bytes into the next), larger ones
SIZES = [256, 257, 320, 447, 448, 449, 512, 513, 640, 641, 1000, 4096, 16383, 70001]


def _letters(n, rng):
    return (97 + rng.integers(0, 26, n)).astype(np.uint8)


def _blanks(n, rng):
    return np.where(rng.random(n) < 0.5, 32, 9).astype(np.uint8)


def _runs(n, rng, k):
    """k runs of punctuation, neighbours different."""
    cuts = np.sort(rng.choice(np.arange(1, n), k - 1, replace=False))
    out = np.empty(n, np.uint8)
    for i, (a, b) in enumerate(zip(np.r_[0, cuts], np.r_[cuts, n])):
        out[a:b] = ord("=-*#"[i % 4])
    return out


KINDS = {
    "letters": _letters,
    "blanks": _blanks,
    "one run": lambda n, rng: np.full(n, ord("="), np.uint8),
    "31 runs": lambda n, rng: _runs(n, rng, 31),
    "32 runs": lambda n, rng: _runs(n, rng, 32),
    "33 runs": lambda n, rng: _runs(n, rng, 33),
    "run and letters": lambda n, rng: np.r_[np.full(n - n // 3, 97, np.uint8), _letters(n // 3, rng)],
    "letters around a run": lambda n, rng: np.r_[_letters(n // 4, rng), np.full(n - 2 * (n // 4), 98, np.uint8), _letters(n // 4, rng)],
}


@pytest.mark.parametrize("name", ["C1", "C3", "C4"])
@pytest.mark.parametrize("kind", list(KINDS))
def test_long_pieces_of_every_shape(name, kind):
    rng = np.random.default_rng(5)
    gv, cv = gpu_vocab(name), cpu_vocab(name)
    for k, n in enumerate(SIZES):
        for pre, suf in ((b"", b""), (b"two words ;\n", b"\nend 12 ")):
            text = np.r_[np.frombuffer(pre, np.uint8), KINDS[kind](n, rng), np.frombuffer(suf, np.uint8)]
            ids, status = gpu_encode(gv, text, offset=k % 5)
            assert status == 0 and same(ids, cv.encode(text, gv.pattern_id)[0]), (kind, n, pre)


def test_many_long_pieces_in_one_call():
    """More long pieces than one stretch of the list holds, of mixed shapes, in a request and in bulk text (over 4 MB)."""
    rng = np.random.default_rng(6)
    gv, cv = gpu_vocab("C3"), cpu_vocab("C3")
    parts, sizes = [], (257, 300, 700, 2500)
    for i in range(900):
        parts += [KINDS[list(KINDS)[i % len(KINDS)]](sizes[i % 4], rng), np.frombuffer(b" x1\n", np.uint8)]
    text = np.concatenate(parts)
    want = cv.encode(text, 0, nthreads=8)[0]
    ids, status = gpu_encode(gv, text)
    assert status == 0 and same(ids, want)
    docs = [text, _letters(3_000_000, rng), text[: text.size // 2]]
    off = np.cumsum([0] + [d.size for d in docs]).astype(np.int64)
    assert off[-1] > 4 << 20
    ids, ids_off, status = gpu_encode_batch(gv, np.concatenate(docs), off)
    assert status == 0
    for d, doc in enumerate(docs):
        assert same(ids[ids_off[d]:ids_off[d + 1]], cv.encode(doc, 0, nthreads=8)[0]), d


@pytest.mark.parametrize("size", [257, 300, 700, 4_672, 4_673])
@pytest.mark.parametrize("name", ["C1", "C4"])
def test_bulk_text_with_more_long_pieces_than_ctas_take(name, size):
    """Beyond eight per CTA (1,184 on 148 SMs) the windows of the pieces go to the whole grid; runs of bytes stay with a CTA."""
    rng = np.random.default_rng(size)
    gv, cv = gpu_vocab(name), cpu_vocab(name)
    n = max(1_200, 4_400_000 // size)
    text = (97 + rng.integers(0, 26, (n, size + 1))).astype(np.uint8)
    text[:, size] = 32
    text[5::97, :size] = ord("=")
    text[7::89, : size // 2] = 97
    ids, status = gpu_encode(gv, text.ravel())
    assert status == 0 and same(ids, cv.encode(text.ravel(), gv.pattern_id, nthreads=8)[0])
