"""Where the kernels change from one way of working to another, against the oracle, exact."""
import random

import numpy as np
import pytest

import workloads as wl
from gpu_util import cpu_vocab, gpu_encode, gpu_encode_batch, gpu_vocab, same, to_dev

pytestmark = pytest.mark.gpu


# the document mask is written 65,536 bytes of text by a CTA: documents that begin at, before and behind such an edge, empty ones
@pytest.mark.parametrize("edge", [65_536, 131_072])
def test_documents_at_the_edges_of_the_mask(edge):
    gv, cv = gpu_vocab("C1"), cpu_vocab("C1")
    text = wl.generate(0, 31, edge + 40_000)
    cuts = sorted({0, 1, 31, 32, 33, edge - 33, edge - 32, edge - 1, edge, edge + 1, edge + 31, edge + 32, text.size - 1})
    off = np.array(cuts[:5] + [cuts[5]] * 3 + cuts[5:] + [text.size] * 2, dtype=np.int64)      # (some documents are empty)
    ids, ioff, status = gpu_encode_batch(gv, text, off)
    assert status == 0
    for d in range(off.size - 1):
        want = cv.encode(text[off[d]:off[d + 1]], 0)[0] if off[d] < off[d + 1] else np.zeros(0, np.int32)
        assert same(ids[ioff[d]:ioff[d + 1]], want), d


# spans: four tokens per thread, 1,024 per block, vector accesses where the buffers allow it
@pytest.mark.parametrize("n", [1, 3, 4, 5, 1023, 1024, 1025, 4097])
@pytest.mark.parametrize("shift", [0, 1])
def test_spans_at_block_edges_and_unaligned_buffers(n, shift):
    import torch
    gv, cv = gpu_vocab("C1"), cpu_vocab("C1")
    ids = cv.encode(wl.generate(1, 5, 20_000), 0)[0][:n]
    size = sum(len(cv.token_bytes(int(i))) for i in ids)
    text = np.frombuffer(b"".join(cv.token_bytes(int(i)) for i in ids), dtype=np.uint8)
    d = torch.zeros(n + shift, dtype=torch.int32, device="cuda")[shift:]
    d.copy_(torch.from_numpy(ids.astype(np.int32)))
    b, c = (torch.full((n + 1 + shift,), -1, dtype=torch.int32, device="cuda")[shift:] for _ in range(2))
    status = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    gv.spans(d, torch.tensor([n], device="cuda"), size, b, c, status)
    torch.cuda.synchronize()
    wb, wc = cv.spans(text, ids)
    assert int(status.item()) == 0 and same(b.cpu().numpy(), wb) and same(c.cpu().numpy(), wc)


# appends: a window of at most 8,192 bytes is one CTA's, text beyond the pinned buffer (256 KB) is copied in front
@pytest.mark.parametrize("context,turn", [(3_000, 7_679), (3_000, 7_680), (3_000, 7_681), (3_000, 7_700), (300_000, 1_500), (2_000, 300_000), (15, 16)])
def test_appends_at_the_limits_of_the_window(context, turn):
    import paper_2607_29678_b200 as tt
    gv, cv = gpu_vocab("C1"), cpu_vocab("C1")
    parts = [wl.generate(0, 7, context), wl.generate(0, 8, turn), wl.generate(1, 9, 200)]
    sess = tt.Session(gv, sum(p.size for p in parts) + 8)
    empty, off, nbytes = sess.records()
    assert empty.numel() == 0 and off.cpu().tolist() == [0] and nbytes == 0
    done = np.zeros(0, np.uint8)
    for part in parts:
        info = sess.append(part)
        done = np.r_[done, part]
        ids, off, nbytes = sess.records()
        want = cv.encode(done, 0)[0]
        assert nbytes == done.size and info["n_tokens"] == want.size and same(ids.cpu().numpy(), want)
        assert same(off.cpu().numpy(), cv.spans(done, want)[0])
    sess.close()


# pageable host buffers: staged whole up to 512 KB, in slices beyond
@pytest.mark.parametrize("n", [1, 4_000, (512 << 10) - 1, 512 << 10, (512 << 10) + 1])
def test_pageable_host_buffers_around_the_staging_limit(n):
    gv, cv = gpu_vocab("C3"), cpu_vocab("C3")
    text = wl.generate(2, 77, n)
    ids = np.full(n + 1, -1, np.int32)
    count = gv.encode_host_into(text, ids)
    assert same(ids[:count], cv.encode(text, 0)[0]) and (ids[count:] == -1).all()


# pattern 1, words with marks: matched on the tile's masks, and on the text where a match leaves the window of 2,304 bytes
@pytest.mark.parametrize("run", [10, 600, 1_150, 2_400, 5_000])
def test_marked_words_that_leave_the_window(run):
    gv, cv = gpu_vocab("C4"), cpu_vocab("C4")
    rng = random.Random(run)
    word = "".join(rng.choice("abcXYZ日'") + "́" * rng.randint(0, 2) for _ in range(run))
    for lead in (0, 700, 1_990, 2_047):
        text = np.frombuffer(("x " * (lead // 2) + " ́" + word + " ende's 12345 \n\n" + "̀" * (run // 4) + word[::-1] + ".").encode(), dtype=np.uint8)
        ids, status = gpu_encode(gv, text)
        assert status == 0 and same(ids, cv.encode(text, 1)[0]), lead


# walks of pattern 1 and 0 over runs of several steps (128 words of 32 bytes each, 120 where neighbours are needed)
@pytest.mark.parametrize("run", [4_095, 8_300, 12_500, 40_000])
@pytest.mark.parametrize("unit", ["7", " ", "/", "\r\n", "'", "ก"])
def test_walks_over_long_runs(run, unit):
    text = np.frombuffer(("日éx'" + unit * (run // len(unit)) + "\n/z 1" + unit * 3_000 + "q́'S").encode(), dtype=np.uint8)
    for name, pattern in (("C1", 0), ("C4", 1)):
        ids, status = gpu_encode(gpu_vocab(name), text)
        assert status == 0 and same(ids, cpu_vocab(name).encode(text, pattern)[0]), (name, pattern)


# pieces of eight, nine, 512 and 513 tokens and an item of more than 2,048 of them on their way out
@pytest.mark.parametrize("n", [8, 9, 512, 513, 2_048, 6_000])
def test_scatter_of_pieces_with_many_tokens(n):
    gv, cv = gpu_vocab("C1"), cpu_vocab("C1")
    rng = np.random.default_rng(n)
    text = np.frombuffer(b"ab " + bytes((97 + rng.integers(0, 26, n)).astype(np.uint8)) + b" cd ef.", dtype=np.uint8)
    text = np.r_[text, np.tile(np.frombuffer("€".encode(), np.uint8), 300), text]
    ids, status = gpu_encode(gv, text)
    assert status == 0 and same(ids, cv.encode(text, 0)[0])
