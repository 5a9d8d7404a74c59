"""Texts of a few tiles, at the tiles' edges and with everything a text can hold, against the oracle."""
import numpy as np
import pytest

import workloads as wl
from gpu_util import cpu_vocab, gpu_encode, gpu_encode_batch, gpu_vocab, same

pytestmark = pytest.mark.gpu

TILE = 2_048
KINDS = [0, 1, 2, 3, 4, 5]


# 4 tiles of 2,048 bytes, counted from the 16-byte boundary below the text
@pytest.mark.parametrize("size", [1, 2, TILE - 1, TILE, TILE + 1, 3 * TILE + 7, 4 * TILE - 16, 4 * TILE - 1, 4 * TILE, 4 * TILE + 1, 5 * TILE])
@pytest.mark.parametrize("offset", [0, 1, 15])
def test_sizes_around_the_edges(size, offset):
    for name, kind in (("C1", 0), ("C4", 2)):
        gv, cv = gpu_vocab(name), cpu_vocab(name)
        text = wl.generate(kind, size, size + 8)[:size]
        ids, status = gpu_encode(gv, text, offset=offset)
        assert status == 0 and same(ids, cv.encode(text, gv.pattern_id)[0])


@pytest.mark.parametrize("pattern", [0, 1, 2, 3])
@pytest.mark.parametrize("kind", KINDS)
def test_every_kind_of_text_and_pattern(pattern, kind):
    gv, cv = gpu_vocab("C1", pattern=pattern), cpu_vocab("C1")
    for chars in (300, 1_500, 2_500):
        text = wl.generate(kind, 40 + chars, chars)
        ids, status = gpu_encode(gv, text)
        assert status == 0 and same(ids, cv.encode(text, pattern)[0]), chars


# pieces of a CTA's size and longer ones, many short pieces, runs that leave the window
@pytest.mark.parametrize("name", ["C1", "C4"])
def test_long_pieces_many_pieces_and_runs(name):
    rng = np.random.default_rng(3)
    gv, cv = gpu_vocab(name), cpu_vocab(name)
    letters = (97 + rng.integers(0, 26, 8_000)).astype(np.uint8)
    texts = [letters, letters[:300], np.r_[letters[:4_700], np.uint8([32]), letters[:2_000]], np.full(8_000, 32, np.uint8), np.full(7_777, 61, np.uint8),
             np.frombuffer(b" ." * 4_000, np.uint8), np.frombuffer(b"7" * 8_000, np.uint8), np.frombuffer(b"\n " * 3_000 + b"x", np.uint8),
             np.frombuffer(b"x's" * 2_000, np.uint8), np.r_[np.full(5_000, 9, np.uint8), letters[:300], np.full(2_000, 10, np.uint8)]]
    for i, text in enumerate(texts):
        ids, status = gpu_encode(gv, text)
        assert status == 0 and same(ids, cv.encode(text, gv.pattern_id)[0]), i


def test_documents_capacity_and_invalid_text():
    gv, cv = gpu_vocab("C1"), cpu_vocab("C1")
    text = wl.generate(0, 5, 7_000)
    off = np.array([0, 0, 1, 33, 2_047, 2_048, 2_049, 5_000, 5_000, 7_000, 7_000], np.int64)
    ids, ioff, status = gpu_encode_batch(gv, text, off)
    want, woff = cv.encode_batch(text, off, 0)
    assert status == 0 and same(ids, want) and same(ioff, woff)
    n = cv.encode(text, 0)[0].size
    assert gpu_encode(gv, text, ids_cap=n)[1] == 0
    ids, status = gpu_encode(gv, text, ids_cap=n - 1)
    assert status == 5 and ids.size == 0
    for at in (0, 2_047, 4_096, 6_999):
        bad = text.copy()
        bad[at] = 0xFF
        ids, status = gpu_encode(gv, bad)
        assert status == 4 and ids.size == 0, at


def test_replayed_from_a_graph_and_beside_other_streams():
    import torch
    gv, cv = gpu_vocab("C3"), cpu_vocab("C3")
    texts = [wl.generate(2, 60 + i, 3_000 + 900 * i) for i in range(4)]
    wants = [cv.encode(t, gv.pattern_id)[0] for t in texts]
    devs, bufs, streams = [torch.from_numpy(t).cuda() for t in texts], [gv.alloc(t.size) for t in texts], [torch.cuda.Stream() for _ in texts]
    torch.cuda.synchronize()
    for _ in range(20):
        for d, b, s in zip(devs, bufs, streams):
            with torch.cuda.stream(s):
                gv.encode(d, b)
    torch.cuda.synchronize()
    for b, w in zip(bufs, wants):
        assert int(b["status"]) == 0 and same(b["ids"][:int(b["count"])].cpu().numpy(), w)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        gv.encode(devs[0], bufs[0])
    other = torch.from_numpy(wl.generate(2, 99, texts[0].size)).cuda()
    devs[0].copy_(other)
    for _ in range(3):
        g.replay()
    torch.cuda.synchronize()
    assert same(bufs[0]["ids"][:int(bufs[0]["count"])].cpu().numpy(), cv.encode(other.cpu().numpy(), gv.pattern_id)[0])


# Entries of ids_off are cleared by the CTAs that have a tile: texts of a few tiles, and one of which some CTAs have none (more tiles than CTAs, two
# to a CTA), with more documents than the CTAs with a tile have threads.
@pytest.mark.parametrize("size", [100, 2_000, 4_000, 8_000, 9_000, 1_300 * TILE])
@pytest.mark.parametrize("n_docs", [1_000, 5_000, 13_000, 400_000])
def test_every_offset_is_zero_on_an_error(size, n_docs):
    import torch
    gv, cv = gpu_vocab("C1"), cpu_vocab("C1")
    text = wl.generate(0, size, size)
    off = np.sort(np.random.default_rng(n_docs).integers(0, size + 1, n_docs + 1))
    off[0], off[-1] = 0, size
    bad, crossed = text.copy(), off.copy()
    bad[size // 2] = 0xFF
    crossed[1] = size + 1
    n = cv.encode_batch(text, off, 0)[0].size
    for t, o, cap, want in ((bad, off, size, 4), (text, off, n - 1, 5), (text, crossed, size, 1), (text, off, n, 0)):
        bufs = gv.alloc(size, max_docs=n_docs)
        bufs["ids"] = bufs["ids"][:cap]
        bufs["ids_off"].fill_(77)
        try:
            gv.encode_batch(torch.from_numpy(t).cuda(), torch.from_numpy(o).cuda(), bufs)
        except Exception as e:
            pytest.fail(str(e))
        torch.cuda.synchronize()
        assert int(bufs["status"]) == want, want
        got = bufs["ids_off"].cpu().numpy()
        if want:
            assert np.flatnonzero(got).size == 0, (want, np.flatnonzero(got).size)
        else:
            assert same(got, cv.encode_batch(text, off, 0)[1])
