"""Batches of very small documents: thousands of them in a stretch of the document mask."""
import numpy as np
import pytest

import workloads as wl
from gpu_util import cpu_vocab, gpu_encode_batch, gpu_vocab, same, to_dev

pytestmark = pytest.mark.gpu


def _expected(cv, text, off, pattern):
    """Documents of at most a few bytes are often the same: each kind is encoded once."""
    seen, ids, ids_off = {}, [], [0]
    raw = text.tobytes()
    for a, b in zip(off[:-1], off[1:]):
        doc = raw[a:b]
        if doc not in seen:
            seen[doc] = cv.encode(np.frombuffer(doc, dtype=np.uint8), pattern)[0] if doc else np.zeros(0, np.int32)
        ids.append(seen[doc])
        ids_off.append(ids_off[-1] + seen[doc].size)
    return np.concatenate(ids), np.array(ids_off)


# 2,048 documents per stretch of 65,536 bytes is where the stretches become shorter: from documents of 32 bytes on
@pytest.mark.parametrize("size,total", [(1, 70_000), (2, 65_535), (3, 65_536), (31, 140_000), (32, 131_072), (33, 140_000), (1, 8_191), (1, 8_193), (7, 262_145)])
def test_documents_of_a_few_bytes(size, total):
    gv, cv = gpu_vocab("C1"), cpu_vocab("C1")
    text = wl.generate(0, size, total)[:total]
    off = np.r_[np.arange(0, total, size), total].astype(np.int64)
    off = np.sort(np.r_[off, off[3:40], np.full(5_000, off[off.size // 2]), [total] * 3])       # some empty ones, many at one place
    ids, ids_off, status = gpu_encode_batch(gv, text, off)
    want, want_off = _expected(cv, text, off, 0)
    assert status == 0 and same(ids_off, want_off) and same(ids, want)


@pytest.mark.parametrize("at", [0, 1, 2_049, 100_000, 199_998, 199_999, 200_000])
def test_a_wrong_offset_among_many_is_found(at):
    gv = gpu_vocab("C1")
    text = wl.generate(0, 1, 200_000)[:200_000]
    off = np.arange(0, 200_001, dtype=np.int64)
    off[at] = {0: 1, 200_000: 199_999}.get(at, off[at] + 2)
    _, ids_off, status = gpu_encode_batch(gv, text, off)
    assert status == 1 and (ids_off == 0).all()


def test_documents_of_one_byte_take_no_longer_than_their_pieces():
    import torch
    gv = gpu_vocab("C2")
    text = wl.generate(0, 3, 400_000)[:400_000]
    d, off = to_dev(text), torch.arange(0, 400_001, dtype=torch.int64, device="cuda")
    bufs, ms = gv.alloc(text.size, max_docs=400_000), []
    for _ in range(12):
        t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda._sleep(100_000)
        t0.record()
        gv.encode_batch(d, off, bufs)
        t1.record()
        torch.cuda.synchronize()
        ms.append(t0.elapsed_time(t1))
    # 0.07 ms; 0.21 where few CTAs read the offsets one by one
    assert int(bufs["status"]) == 0 and np.median(ms) < 0.13, ms
