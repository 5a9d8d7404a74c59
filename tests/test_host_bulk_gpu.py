"""Host calls around the limit of bulk text (4 MB), where ids go to a pinned buffer by one copy instead of being written there."""
import numpy as np
import pytest

import workloads as wl
from gpu_util import cpu_vocab, gpu_vocab, same

pytestmark = pytest.mark.gpu

LIMIT = 2_048 * 2_048


@pytest.mark.parametrize("pinned_in", [False, True])
@pytest.mark.parametrize("n", [LIMIT - 16, LIMIT - 15, LIMIT - 14, LIMIT, LIMIT + 1, 9_000_000])
def test_pinned_ids_around_the_limit(n, pinned_in):
    import torch
    import paper_2607_29678_b200 as tt
    gv, cv = gpu_vocab("C3"), cpu_vocab("C3")
    text = wl.generate(2, 5, n)[:n]
    want = cv.encode(text, 0, nthreads=8)[0]
    t = torch.from_numpy(text.copy())
    t = t.pin_memory() if pinned_in else t
    ids = torch.full((want.size + 3,), -1, dtype=torch.int32).pin_memory()
    count = gv.encode_host_into(t, ids)
    assert count == want.size and same(ids[:count].numpy(), want) and (ids[count:] == -1).all()
    small = torch.full((want.size,), -1, dtype=torch.int32).pin_memory()
    with pytest.raises(tt.TokTierError) as e:
        gv.encode_host_into(t, small[:-1])
    assert e.value.code == tt.TT_ERR_CAPACITY and (small == -1).all()


def test_pinned_ids_of_bulk_text_take_no_longer_than_pageable_ones():
    import time
    import torch
    gv = gpu_vocab("C3")
    t = torch.from_numpy(wl.generate(2, 6, 8_000_000)).pin_memory()

    def per_call(ids):
        ms = []
        for _ in range(9):
            t0 = time.perf_counter()
            gv.encode_host_into(t, ids)
            ms.append(time.perf_counter() - t0)
        return np.median(ms[2:])

    pageable, pinned = per_call(torch.zeros(4_000_000, dtype=torch.int32)), per_call(torch.zeros(4_000_000, dtype=torch.int32).pin_memory())
    # 2.7 times where the kernel wrote to the pinned buffer itself
    assert pinned < 1.3 * pageable, (pinned, pageable)
