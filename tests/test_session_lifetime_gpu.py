"""Sessions beside other work on the device: what their creation, copies and end do to other streams, captures and memory."""
import ctypes
import threading

import numpy as np
import pytest

import workloads as wl
from gpu_util import cpu_vocab, gpu_vocab, same

pytestmark = pytest.mark.gpu


def _during_a_capture_of_another_thread(action):
    """Runs action() while a capture (thread-local mode) is under way here; the graph has to come out whole."""
    import torch
    x = torch.zeros(1024, device="cuda")
    torch.cuda.synchronize()
    go, done, errors = threading.Event(), threading.Event(), []

    def other():
        go.wait()
        try:
            action()
        except Exception as e:
            errors.append(e)
        done.set()

    t = threading.Thread(target=other)
    t.start()
    graph = torch.cuda.CUDAGraph()
    try:
        with torch.cuda.graph(graph, stream=torch.cuda.Stream(), capture_error_mode="thread_local"):
            x.add_(1)
            go.set()
            done.wait(60)
            x.add_(1)
    finally:
        go.set()
        t.join()
    graph.replay()
    torch.cuda.synchronize()
    assert not errors and bool((x == 2).all())


@pytest.mark.parametrize("copied", [False, True])
def test_the_end_of_a_session_leaves_other_captures_alone(copied):
    import paper_2607_29678_b200 as tt
    sess = tt.Session(gpu_vocab("C1"), 50_000)
    sess.append(wl.generate(0, 1, 5_000))
    if copied:
        sess.records()
    _during_a_capture_of_another_thread(sess.close)


def test_a_copy_on_its_way_survives_the_session():
    """The memory of a freed session goes to the next one, but not before the copies out of it are through."""
    import torch
    import paper_2607_29678_b200 as tt
    gv, cv = gpu_vocab("C1"), cpu_vocab("C1")
    text = wl.generate(0, 2, 20_000)
    want = cv.encode(text, 0)[0]
    sess = tt.Session(gv, 30_000)
    sess.append(text)
    outs = []
    for stream in (torch.cuda.Stream(), torch.cuda.Stream()):
        ids = torch.zeros(want.size, dtype=torch.int32, device="cuda")
        off = torch.zeros(want.size + 1, dtype=torch.int32, device="cuda")
        count = torch.zeros(1, dtype=torch.int64, device="cuda")
        torch.cuda.current_stream().synchronize()
        with torch.cuda.stream(stream):
            torch.cuda._sleep(40_000_000)
            tt._check(tt.lib().tt_session_copy(sess._h, ids.data_ptr(), want.size, off.data_ptr(), count.data_ptr(), stream.cuda_stream), "tt_session_copy")
        outs.append((ids, off, count))
    sess.close()
    other = tt.Session(gv, 30_000)
    other.append(wl.generate(1, 3, 25_000))
    torch.cuda.synchronize()
    for ids, off, count in outs:
        assert int(count) == want.size and same(ids.cpu().numpy(), want) and same(off.cpu().numpy(), cv.spans(text, want)[0])
    other.close()


def test_the_view_of_an_empty_session_leaves_other_captures_alone():
    import paper_2607_29678_b200 as tt
    sess = tt.Session(gpu_vocab("C1"), 50_000)
    pointers = [ctypes.c_void_p() for _ in range(3)]
    size = ctypes.c_size_t(7)
    _during_a_capture_of_another_thread(lambda: tt._check(tt.lib().tt_session_view(sess._h, *map(ctypes.byref, pointers), ctypes.byref(size)), "tt_session_view"))
    assert size.value == 0 and all(p.value for p in pointers)
    sess.close()


@pytest.mark.parametrize("failed", [False, True])
def test_a_copy_of_an_empty_session_can_be_captured(failed):
    """Also after an append that failed and left the session empty."""
    import torch
    import paper_2607_29678_b200 as tt
    sess = tt.Session(gpu_vocab("C1"), 50_000)
    if failed:
        with pytest.raises(tt.TokTierError):
            sess.append(np.frombuffer(b"abc \xff def", dtype=np.uint8))
    off = torch.full((4,), 7, dtype=torch.int32, device="cuda")
    count = torch.full((1,), 7, dtype=torch.int64, device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, capture_error_mode="thread_local"):
        tt._check(tt.lib().tt_session_copy(sess._h, None, 3, off.data_ptr(), count.data_ptr(), torch.cuda.current_stream().cuda_stream), "tt_session_copy")
    graph.replay()
    torch.cuda.synchronize()
    assert int(count) == 0 and off.tolist() == [0, 7, 7, 7]
    ids, offsets, size = sess.records()
    assert ids.numel() == 0 and offsets.tolist() == [0] and size == 0
    sess.close()


def test_a_captured_copy_takes_what_the_session_has_when_it_runs():
    import torch
    import paper_2607_29678_b200 as tt
    gv, cv = gpu_vocab("C1"), cpu_vocab("C1")
    parts = [wl.generate(0, 4, 500), wl.generate(0, 5, 4_000)]
    sess = tt.Session(gv, 10_000)
    sess.append(parts[0])
    cap = 1_000
    ids = torch.zeros(cap, dtype=torch.int32, device="cuda")
    off = torch.zeros(cap + 1, dtype=torch.int32, device="cuda")
    count = torch.zeros(1, dtype=torch.int64, device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, capture_error_mode="thread_local"):
        tt._check(tt.lib().tt_session_copy(sess._h, ids.data_ptr(), cap, off.data_ptr(), count.data_ptr(), torch.cuda.current_stream().cuda_stream), "tt_session_copy")
    text = np.zeros(0, np.uint8)
    for part in [None] + parts[1:]:
        if part is not None:
            sess.append(part)
        text = np.r_[text, parts[0] if part is None else part]
        graph.replay()
        torch.cuda.synchronize()
        want, n = cv.encode(text, 0)[0], int(count)
        k = min(n, cap)
        assert n == want.size and same(ids[:k].cpu().numpy(), want[:k]) and same(off[:k + 1].cpu().numpy(), cv.spans(text, want)[0][:k + 1])
    assert n > cap
    sess.close()


def _free():
    import torch
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def _own_vocab():
    import paper_2607_29678_b200 as tt
    return tt.Vocab(*wl.load_vocab(wl.CONFIGS["C1"]), 0)


def test_a_larger_session_finds_a_place_among_the_kept_ones():
    """Eight small sessions have ended; a larger one leaves its memory to the next one of its size all the same."""
    import paper_2607_29678_b200 as tt
    v = _own_vocab()
    small = [tt.Session(v, 1_000_000) for _ in range(8)]
    for s in small:
        s.close()
    tt.Session(v, 6_000_000).close()                         # (about 45 bytes of device memory per byte: more than 4 times a small one's)
    before = _free()
    large = tt.Session(v, 6_000_000)
    assert _free() == before                                  # nothing was allocated for it
    large.append(wl.generate(0, 1, 3_000))
    large.close()
    assert _free() == before
    v.close()
    assert _free() > before + (200 << 20)


@pytest.mark.parametrize("what", ["session", "host call"])
def test_kept_memory_gives_way_when_none_is_left(what):
    import torch
    import paper_2607_29678_b200 as tt
    v, cv = _own_vocab(), cpu_vocab("C1")
    text = wl.generate(0, 1, 8_000_000 if what == "host call" else 3_000)
    want = cv.encode(text, 0, nthreads=8)[0]
    kept = [tt.Session(v, 1_300_000) for _ in range(8)]       # about 60 MB each
    for s in kept:
        s.close()
    hold = torch.empty(_free() - (150 << 20), dtype=torch.uint8, device="cuda")      # 150 MB are left, and what the vocabulary keeps
    try:
        if what == "session":
            sess = tt.Session(v, 8_000_000)                   # about 380 MB
            assert sess.append(text)["n_tokens"] == want.size
            sess.close()
        else:
            assert same(v.encode_host(text), want)            # about 360 MB of device memory
    finally:
        del hold
        torch.cuda.empty_cache()
        v.close()
