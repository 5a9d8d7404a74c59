"""Caller ids in orders other than bytes first and results by rank: bytes in any order, results from any number on, no order at all."""
import numpy as np
import pytest

import oracle
import workloads as wl
from gpu_util import gpu_encode, gpu_encode_batch, same

pytestmark = pytest.mark.gpu


def _ids(how, n):
    """Caller id of every internal token: 256 bytes, then the results."""
    rng = np.random.default_rng(3)
    ids = np.arange(n)
    if how == "bytes permuted":
        ids[:256] = rng.permutation(256)
    elif how == "bytes last":
        ids = np.r_[np.arange(n - 256, n), np.arange(n - 256)]
    elif how == "results far off":
        ids[:256], ids[256:] = 5 + 2 * rng.permutation(256), 100_000 + np.arange(n - 256)
    elif how == "two results swapped":
        ids[[n - 1, n - 2]] = ids[[n - 2, n - 1]]
    elif how == "no order":
        ids = rng.permutation(n)
    return ids.astype(np.int32)


@pytest.mark.parametrize("n_merges", [0, 1, 4_096])
@pytest.mark.parametrize("how", ["bytes first", "bytes permuted", "bytes last", "results far off", "two results swapped", "no order"])
def test_ids_in_other_orders(how, n_merges):
    import paper_2607_29678_b200 as tt
    if how == "two results swapped" and n_merges < 2:
        pytest.skip("needs two results")
    merges, byte_map = wl.load_vocab(wl.CONFIGS["C1"])
    ids = _ids(how, 256 + n_merges)
    internal = np.zeros(int(merges.max()) + 1, np.int64)
    internal[byte_map] = np.arange(256)
    internal[merges[:, 2]] = 256 + np.arange(len(merges))
    m, bm = ids[internal[merges[:n_merges]]].reshape(-1, 3), ids[:256]
    gv, cv = tt.Vocab(m, bm, 0), oracle.Vocab(m, bm)
    for kind, n in ((1, 30_000), (5, 40_000), (3, 150_000)):
        text = wl.generate(kind, 2, n)
        got, status = gpu_encode(gv, text)
        assert status == 0 and same(got, cv.encode(text, 0, nthreads=8)[0]), kind
    text = wl.generate(1, 4, 4_300_000)                       # bulk text
    off = np.array([0, text.size], dtype=np.int64)
    got, ids_off, status = gpu_encode_batch(gv, text, off)
    assert status == 0 and same(got, cv.encode(text, 0, nthreads=8)[0])
    gv.close()
