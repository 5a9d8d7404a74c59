"""Pattern 1: words whose last sure piece start lies far before the tile's window are matched over the text, all lanes of a
warp side by side."""
import numpy as np
import pytest

from gpu_util import cpu_vocab, gpu_encode_batch, gpu_vocab, same, to_dev

pytestmark = pytest.mark.gpu

TEXTS = {"suffixes": "x'd", "suffix chain": "'s", "marks": "́", "upper after caseless": "日A"}


@pytest.mark.parametrize("lead", ["", "\n", "a 1. "])
@pytest.mark.parametrize("name", list(TEXTS))
def test_matches_far_from_a_sure_start(name, lead):
    import torch
    gv, cv = gpu_vocab("C4"), cpu_vocab("C4")
    text = np.frombuffer((lead + TEXTS[name] * (15_000 // len(TEXTS[name].encode())) + " end").encode(), dtype=np.uint8)
    want = cv.encode(text, 1)[0]
    d, bufs, ms = to_dev(text), gv.alloc(text.size), []
    for _ in range(5):
        t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        t0.record()
        gv.encode(d, bufs, length=text.size)
        t1.record()
        torch.cuda.synchronize()
        ms.append(t0.elapsed_time(t1))
    assert int(bufs["status"]) == 0 and same(bufs["ids"][:int(bufs["count"])].cpu().numpy(), want)
    # about 2.5 ms for 15 KB with the lanes of a warp together, 35 to 80 ms one after the other
    assert min(ms) < 12.0, ms


def test_far_matches_end_with_their_document():
    gv, cv = gpu_vocab("C4"), cpu_vocab("C4")
    docs = [np.frombuffer((TEXTS[k] * n + tail).encode(), dtype=np.uint8) for k in TEXTS for n, tail in ((1_500, ""), (700, "\n"), (2_000, "z"))]
    off = np.cumsum([0] + [d.size for d in docs]).astype(np.int64)
    ids, ids_off, status = gpu_encode_batch(gv, np.concatenate(docs), off)
    assert status == 0
    for i, doc in enumerate(docs):
        assert same(ids[ids_off[i]:ids_off[i + 1]], cv.encode(doc, 1)[0]), i
