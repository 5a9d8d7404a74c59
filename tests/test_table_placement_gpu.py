"""Whole-piece table: entries whose hashes collide have to find a place, whatever their number."""
import numpy as np
import pytest

import oracle
from gpu_util import gpu_encode, same

pytestmark = pytest.mark.gpu

# Entries of one length whose key words have one sum under the table's first multipliers: they share both buckets.  A bucket of the
# table for 9 to 24 bytes holds one entry, one of the table for up to 8 bytes two.
ALIKE = {
    "two of 9 bytes": [b"fgyamdeya", b"xtxopdeyv"],
    "three of 9 bytes": [b"fgyamdeya", b"xtxopdeyv", b"tvqwvspkh"],
    "three others": [b"otfvukoys", b"acggzxqvr", b"ltfbjlqhk"],
    "four of 8 bytes": [b"vcegeuwp", b"vcvieuhf", b"vtouefur", b"ejafthsr"],
    "eleven of 8 bytes": [b"vcegeuwp", b"vcvieuhf", b"vtouefur", b"ejafthsr", b"ergetphs", b"ejrhthdh", b"erostppp", b"erwytpxe", b"ezdytxtd", b"ejrpthdp", b"vtggefmu"],
}
ALIKE["all"] = [s for k in ("three of 9 bytes", "three others", "eleven of 8 bytes") for s in ALIKE[k]]


def _vocabulary(strings):
    """Merges that build every string from the left."""
    merges, ids = [], {}
    for s in strings:
        cur = s[0]
        for ch in s[1:]:
            if (cur, ch) not in ids:
                ids[cur, ch] = 256 + len(merges)
                merges.append((cur, ch, 256 + len(merges)))
            cur = ids[cur, ch]
    return np.array(merges, dtype=np.int32)


@pytest.mark.parametrize("ignore_merges", [False, True])
@pytest.mark.parametrize("name", list(ALIKE))
def test_entries_that_share_both_buckets(name, ignore_merges):
    import paper_2607_29678_b200 as tt
    strings = ALIKE[name]
    merges = _vocabulary(strings)
    gv, cv = tt.Vocab(merges, None, 0, ignore_merges=ignore_merges), oracle.Vocab(merges, ignore_merges=ignore_merges)
    assert gv.table_entries() >= len(strings)
    text = np.frombuffer(b"".join(s + b"\n" + s[:-1] + b"." + s + s for s in strings) * 3, dtype=np.uint8)
    ids, status = gpu_encode(gv, text)
    assert status == 0 and same(ids, cv.encode(text, 0)[0])
    gv.close()
