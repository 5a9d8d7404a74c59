"""What the first kernel, the merges and the scatter of bulk text hand each other, against the oracle."""
import numpy as np
import pytest

import workloads as wl
from gpu_util import cpu_vocab, gpu_encode, gpu_encode_batch, gpu_vocab, same

pytestmark = pytest.mark.gpu


# pieces of so many tokens that their number does not fit the record (2^20 - 1 and more), and fewer; starts all over the tile
@pytest.mark.parametrize("tokens", [1_048_573, 1_048_574, 1_048_575, 2_200_000])
@pytest.mark.parametrize("before", [0, 1, 2_040])
def test_a_piece_of_more_tokens_than_the_record_holds(tokens, before):
    gv, cv = gpu_vocab("C1"), cpu_vocab("C1")
    # control characters: one punctuation piece with the line feed behind it; no merge knows them (checked below), so a token per byte
    long = np.tile(np.uint8([1, 2, 3]), tokens // 3 + 1)[:tokens]
    assert cv.encode(long[:3_000], 0)[0].size == 3_000
    text = np.r_[np.full(before, 97, np.uint8), np.uint8([10]), long, np.frombuffer(b"\nand so on.\n", np.uint8), wl.generate(0, 3, 4_300_000)]
    ids, status = gpu_encode(gv, text)
    assert status == 0 and same(ids, cv.encode(text, 0, nthreads=8)[0])


# groups of 32 pieces: none, one and all of them merged, of up to eight tokens and of more
@pytest.mark.parametrize("every", [1, 2, 31, 32, 33, 200])
@pytest.mark.parametrize("size", [9, 14, 90])
def test_merged_pieces_among_settled_ones(every, size):
    rng = np.random.default_rng(every * 100 + size)
    gv, cv = gpu_vocab("C3"), cpu_vocab("C3")
    settled = b" the" * (every - 1)
    words = (97 + rng.integers(0, 26, (4_400_000 // (len(settled) + size + 1), size))).astype(np.uint8)
    text = np.concatenate([np.r_[np.frombuffer(settled, np.uint8), np.uint8([32]), w] for w in words])
    ids, status = gpu_encode(gv, text)
    assert status == 0 and same(ids, cv.encode(text, 0, nthreads=8)[0])


# runs of neighbouring tiles are one CTA's, which keeps the end of the tile before: constructs of every kind across every edge,
# at every place, in one text and in documents
SNIPPETS = [b"it's we'll they've I'd ", b" 1234567890123 ", b"   \n\n  \r\n   x", b"!!!\n\n??? \n", "é ñ日本語 x  y ".encode(), b"don't" * 3, b" '' 's 't 'll",
            b"a" * 70, b" " * 300 + b"x", b"7" * 400]


# (on 148 SMs the CTAs take runs of 1, 2, 2, 3, 5 and 8 tiles)
@pytest.mark.parametrize("pattern,megabytes,docs", [(p, m, d) for p in (0, 1, 2, 3) for m, d in ((5, 0), (14, 0), (14, 3_000), (26, 0))] +
                         [(0, 44, 0), (2, 44, 5_000), (3, 44, 0), (2, 62, 0), (0, 103, 0), (0, 103, 9_000)])
def test_constructs_across_the_edges_of_neighbouring_tiles(pattern, megabytes, docs):
    rng = np.random.default_rng(megabytes + pattern)
    gv, cv = gpu_vocab("C1", pattern=pattern), cpu_vocab("C1")
    filler = wl.generate(0, 17, megabytes * 1_000_000)
    at = 2_048
    while at + 2_048 < filler.size:                                    # a construct across every edge, one byte further each time
        s = np.frombuffer(SNIPPETS[int(rng.integers(len(SNIPPETS)))], np.uint8)
        from_ = at - int(rng.integers(0, s.size + 1))
        filler[from_:from_ + s.size] = s
        at += 2_048
    if not docs:
        ids, status = gpu_encode(gv, filler)
        assert status == 0 and same(ids, cv.encode(filler, pattern, nthreads=8)[0])
        return
    cuts = np.unique(rng.integers(1, filler.size, docs))
    cuts = cuts[(filler[cuts] & 0xC0) != 0x80]
    off = np.r_[0, cuts, filler.size].astype(np.int64)
    ids, ioff, status = gpu_encode_batch(gv, filler, off)
    want, woff = cv.encode_batch(filler, off, pattern, nthreads=8)
    assert status == 0 and same(ids, want) and same(ioff, woff)


# a tile whose first word the CTA has kept from the tile before does not look at it again: bytes that are no UTF-8, and documents that begin
# inside a character, at every place around the edges of a run's tiles
@pytest.mark.parametrize("pattern", [0, 2])
def test_invalid_text_around_the_edges_of_neighbouring_tiles(pattern):
    import torch
    gv = gpu_vocab("C1", pattern=pattern)
    text = wl.generate(0, 23, 44_000_000)                              # ASCII; runs of three tiles on 148 SMs
    d, bufs = torch.from_numpy(text).cuda(), gv.alloc(text.size, max_docs=2)
    places = [2_048 * t + o for t in (1, 2, 3, 4, 5, 6, 21_482, 21_483, 21_484) for o in (-33, -32, -1, 0, 1, 31, 32, 33)]

    def statuses(bytes_, off):
        found = torch.zeros(len(places), dtype=torch.int32, device="cuda")
        for i, at in enumerate(places):
            kept = d[at:at + len(bytes_)].clone()
            d[at:at + len(bytes_)] = torch.tensor(list(bytes_), dtype=torch.uint8, device="cuda")
            if off is None:
                gv.encode(d, bufs)
            else:
                gv.encode_batch(d, torch.tensor([0, at + off, text.size], dtype=torch.int64, device="cuda"), bufs)
            found[i] = bufs["status"][0]
            d[at:at + len(bytes_)] = kept
        return found.cpu().numpy()

    assert d.data_ptr() % 16 == 0 and 2_048 * 21_484 + 40 < text.size
    assert (statuses(b"\xff", None) == 4).all()
    assert (statuses(b"\x80", None) == 4).all()
    assert (statuses(b"\xe3a", None) == 4).all()                       # a lead byte without the rest
    assert (statuses(b"\xc3\xa9", None) == 0).all()
    assert (statuses(b"\xc3\xa9", 1) == 4).all()                       # a document that begins with a continuation byte
    assert (statuses(b"\xc3\xa9", 0) == 0).all()
