"""Added tokens by the thousand: the entries a byte is compared with are read several at a time."""
import numpy as np
import pytest

import oracle
import workloads as wl
from gpu_util import same, to_dev

pytestmark = pytest.mark.gpu


def _vocab(literals):
    import paper_2607_29678_b200 as tt
    merges, byte_map = wl.load_vocab(wl.CONFIGS["C1"])
    gv, ids = tt.Vocab(merges, byte_map, 0), [500_000 + k for k in range(len(literals))]
    gv.add_literals(literals, ids)
    return gv, oracle.Vocab(merges, byte_map), ids


# eight entries are looked at together; literals of every length up to the number of them, each a prefix of the next
@pytest.mark.parametrize("n", [1, 7, 8, 9, 15, 16, 17, 200])
def test_the_longest_of_many_prefixes(n):
    import torch
    literals = [("<|" + "ab" * n)[: k + 1] for k in range(n)]
    gv, cv, ids = _vocab(literals)
    rng = np.random.default_rng(n)
    s = " ".join(("<|" + "ab" * n)[: int(k)] + "x" * int(k % 3) for k in rng.integers(1, n + 6, 400)) + literals[-1]
    text = np.frombuffer(s.encode(), dtype=np.uint8)
    d, bufs = to_dev(text, n % 16), gv.alloc(text.size)
    gv.encode_added(d, bufs, length=text.size)
    torch.cuda.synchronize()
    assert int(bufs["status"]) == 0
    assert same(bufs["ids"][:int(bufs["count"])].cpu().numpy(), oracle.encode_added(cv, text, 0, literals, ids))


@pytest.mark.parametrize("shift", [0, 3])
def test_the_second_byte_and_the_ninth(shift):
    """A byte is left alone where no literal has the byte behind it, but for literals of one byte; the first eight bytes are compared at
    once.  The blob may begin anywhere in the caller's array."""
    import torch
    import paper_2607_29678_b200 as tt
    rng = np.random.default_rng(shift)
    for literals in (["<|", "<"], ["<|", "<", "abcdefgh", "abcdefghi", "abcdefgj", "|x", "hi", "e\0", "i"], ["<|", "ab", "abcdefgh", "abcdefghij", "hiab", "bcd", "efg", "eee", "|<|<|<|<|"], ["<|", "ab"], ["abcdefgh", "abcdefghi", "abcdefghj", "abcdefg"], ["e"], ["\0", "e\0"], ["<|abcde", "<|abcdef", "<|abcdefg", "|"]):
        merges, byte_map = wl.load_vocab(wl.CONFIGS["C1"])
        gv, cv, ids = tt.Vocab(merges, byte_map, 0), oracle.Vocab(merges, byte_map), [600_000 + k for k in range(len(literals))]
        blob = np.frombuffer(("xyz"[:shift] + "".join(literals)).encode(), dtype=np.uint8)
        off = (shift + np.cumsum([0] + [len(x) for x in literals])).astype(np.uint32)
        idv = np.array(ids, np.int32)
        tt._check(tt.lib().tt_vocab_add_literals(gv._h, blob.ctypes.data, off.ctypes.data, idv.ctypes.data, len(literals)), "tt_vocab_add_literals")
        parts = literals + [x[:-1] for x in literals] + ["<", "|", "a", "b", "e", " ", "h", "i", "\0"]
        text = np.frombuffer("".join(parts[int(k)] for k in rng.integers(0, len(parts), 6_000)).encode(), dtype=np.uint8)
        for t in (text, text[: 1], text[-1:]):
            d, bufs = to_dev(t, shift), gv.alloc(t.size)
            gv.encode_added(d, bufs, length=t.size)
            torch.cuda.synchronize()
            assert int(bufs["status"]) == 0
            assert same(bufs["ids"][:int(bufs["count"])].cpu().numpy(), oracle.encode_added(cv, t, 0, literals, ids)), literals


@pytest.mark.parametrize("unit,limit_ms", [("<", 1.09), ("<|r_0|>", 0.88)])
def test_two_thousand_literals_that_begin_alike(unit, limit_ms):
    """The bound is what a thread per byte took, comparing entry by entry (3.3 and 1.25 ms with a thread per 16 bytes)."""
    import torch
    literals = [f"<|r_{i}|>" for i in range(2_000)]
    gv, cv, ids = _vocab(literals)
    text = np.frombuffer((unit * (300_000 // len(unit))).encode(), dtype=np.uint8)
    d, bufs, ms = to_dev(text), gv.alloc(text.size), []
    for _ in range(9):
        t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda._sleep(100_000)
        t0.record()
        gv.encode_added(d, bufs, length=text.size)
        t1.record()
        torch.cuda.synchronize()
        ms.append(t0.elapsed_time(t1))
    got = bufs["ids"][:int(bufs["count"])].cpu().numpy()
    want = np.full(text.size // len(unit), ids[0]) if len(unit) > 1 else cv.encode(text, 0)[0]
    assert int(bufs["status"]) == 0 and same(got, want)
    assert np.median(ms) < limit_ms, ms
