"""Literals that cannot overlap (none holds the byte another begins with): one kernel writes their masks, 2,048 bytes of text to a CTA."""
import numpy as np
import pytest

import oracle
import workloads as wl
from gpu_util import to_dev, same

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lengths", [[1], [2, 5], [4, 8, 9, 33], [255], [1, 16, 17, 100, 254, 255]])
@pytest.mark.parametrize("offset", [0, 3])
@pytest.mark.parametrize("pattern", [0, 1, 3])
def test_literals_across_the_edges(lengths, offset, pattern):
    import torch
    import paper_2607_29678_b200 as tt
    merges, byte_map = wl.load_vocab(wl.CONFIGS["C1"])
    cv, gv = oracle.Vocab(merges, byte_map), tt.Vocab(merges, byte_map, pattern)
    lits = ["\x01" + "ab|>"[:n - 1] + "x" * (n - 5) if n > 5 else ("\x01" + "ab|>")[:n] for n in lengths]
    ids = [700_000 + k for k in range(len(lits))]
    gv.add_literals(lits, ids)
    rng = np.random.default_rng(len(lits))
    text = wl.generate(0, 21, 3 * 65_536)
    raw = [np.frombuffer(x.encode(), np.uint8) for x in lits]
    for edge in range(2_048, text.size - 2_048, 2_048):                 # so that they end at, cross and begin behind every edge
        x = raw[int(rng.integers(len(raw)))]
        at = edge - offset - int(rng.integers(0, x.size + 2)) + int(rng.integers(0, 2))
        text[at:at + x.size] = x
    text[-raw[0].size:] = raw[0]
    text[:raw[-1].size] = raw[-1]
    for part in (text, text[:2_047], text[:4_096], text[:1]):
        d, bufs = to_dev(part, offset), gv.alloc(part.size)
        gv.encode_added(d, bufs, length=part.size)
        torch.cuda.synchronize()
        want = oracle.encode_added(cv, part, pattern, lits, ids)
        assert int(bufs["status"]) == 0 and same(bufs["ids"][:int(bufs["count"])].cpu().numpy(), want), part.size


def test_many_of_them_side_by_side():
    import torch
    import paper_2607_29678_b200 as tt
    merges, byte_map = wl.load_vocab(wl.CONFIGS["C1"])
    cv, gv = oracle.Vocab(merges, byte_map), tt.Vocab(merges, byte_map, 0)
    lits = ["<%d>" % k for k in range(300)]
    ids = [600_000 + k for k in range(300)]
    gv.add_literals(lits, ids)
    rng = np.random.default_rng(1)
    text = np.frombuffer("".join(lits[int(k)] + ("a" if k % 7 == 0 else "") for k in rng.integers(0, 300, 12_000)).encode(), np.uint8)
    d, bufs = to_dev(text), gv.alloc(text.size)
    gv.encode_added(d, bufs, length=text.size)
    torch.cuda.synchronize()
    want = oracle.encode_added(cv, text, 0, lits, ids)
    assert int(bufs["status"]) == 0 and same(bufs["ids"][:int(bufs["count"])].cpu().numpy(), want)
