"""The scatter kernel on records that contradict each other: a tile's pieces add up to more tokens than its count says.  No call
leaves such records, so the kernel is launched here on records made by hand."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_29678_b200", "csrc")
SOURCE = r"""
#include "tt_bpe.cuh"
extern "C" int run(int ntiles, const u32* tile_cnt, const u32* tile_tok, const u16* off16, const u32* piece_cnt, const int32_t* stage,
                   int32_t* ids_out, long long* count_out, int32_t* status_out, u32 cap, TTHeader* hdr) {
    ScatterParams S = {};
    S.shift = 0; S.hi = (long long)ntiles * TT_TILE_BYTES; S.ntiles = ntiles; S.tile_cnt = tile_cnt; S.tile_tok = tile_tok; S.piece_off16 = off16;
    S.ids_cap = cap; S.piece_cnt = piece_cnt; S.stage = stage; S.hdr = hdr; S.epoch = 1;
    S.ids_out = ids_out; S.count_out = count_out; S.status_out = status_out;
    k_scatter<SCATTER_CTAS><<<ntiles, BPE_THREADS>>>(S);
    return (int)cudaDeviceSynchronize();
}
"""
TILE = 2048
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")


@pytest.fixture(scope="module")
def scatter(tmp_path_factory):
    if not shutil.which(NVCC):
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("scatter")
    (d / "scatter.cu").write_text(SOURCE)
    subprocess.check_call([NVCC, "-gencode", "arch=compute_100a,code=sm_100a", "-O1", "-std=c++17", "-I", CSRC, "-shared", "-Xcompiler", "-fPIC",
                           "-o", str(d / "scatter.so"), str(d / "scatter.cu")])
    return ctypes.CDLL(str(d / "scatter.so")).run


# tokens per piece (1: an id of its own; more: staged) and how many tokens fewer the tile's record says
@pytest.mark.parametrize("pieces,short", [([1] * 10, 0), ([1] * 10, 4), ([1] * 600, 1), ([2, 8, 1] * 100, 5), ([9, 1, 40] * 30, 7), ([1] * 10, 10)])
def test_nothing_is_written_beyond_the_total(scatter, pieces, short):
    import torch
    ntiles = 2
    cnt, off, pos = np.zeros((ntiles, TILE), np.int32), np.zeros((ntiles, TILE), np.uint16), 0
    stage, want = np.zeros(ntiles * TILE, np.int32), []
    for i, n in enumerate(pieces):
        cnt[0, i], off[0, i] = (7_000 + i if n == 1 else -n), pos
        stage[pos:pos + n] = 100 * i + np.arange(n)
        want += [7_000 + i] if n == 1 else list(100 * i + np.arange(n))
        pos += n + 1
    assert pos <= TILE
    dev = [torch.from_numpy(a).cuda() for a in (np.array([len(pieces), 0], np.int32), np.array([len(want) - short, 0], np.int32), off.view(np.int16).ravel(), cnt.ravel(), stage)]
    total = len(want) - short
    ids = torch.full((4 * TILE,), -1, dtype=torch.int32, device="cuda")        # more than the pieces can add up to
    count, status, hdr = torch.full((1,), -1, dtype=torch.int64, device="cuda"), torch.full((1,), -1, dtype=torch.int32, device="cuda"), torch.zeros(256, dtype=torch.uint8, device="cuda")
    p = [ctypes.c_void_p(t.data_ptr()) for t in dev + [ids, count, status]]
    torch.cuda.synchronize()
    assert scatter(ntiles, *p, total, ctypes.c_void_p(hdr.data_ptr())) == 0
    got = ids.cpu().numpy()
    assert int(count) == total and int(status) == 0
    assert (got[total:] == -1).all()
    if short == 0:
        assert (got[:total] == want).all()
