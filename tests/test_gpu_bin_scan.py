"""The scan of the binning's tile counts at the edges of its block of 4096 tiles, and the
count and scatter passes at each chunk size, against the oracle's lists."""
from __future__ import annotations

import numpy as np
import pytest

from gpu_util import native, torch_cuda
from oracle import oracle as O
from test_gpu_parity import bin_case_records, gpu_bin, gpu_lists, rec_to_gpu

pytestmark = pytest.mark.gpu


def length_class(lens):
    """Lengths below 8 by themselves, then eight classes to the octave."""
    e = np.floor(np.log2(np.maximum(lens, 1))).astype(np.int64)
    return np.where(lens < 8, lens, 8 * (e - 2) + ((lens >> np.maximum(e - 3, 0)) & 7))


@pytest.mark.parametrize("case", [
    # V, n, W, H, B, max radius
    (1, 40, 8, 8, 8, 3),            # one tile
    (1, 700, 512, 504, 8, 40),      # 4032 tiles
    (1, 700, 512, 512, 8, 40),      # 4096: one whole block
    (1, 700, 514, 512, 8, 40),      # 4160: two blocks
    (3, 257, 512, 512, 8, 90),      # three blocks
    (1, 300, 512, 512, 8, 34),      # rects around the 64 tiles of a mask
    (1, 60, 512, 512, 8, 900),      # rects of the whole view: 32 runs of 128 tiles
    (1, 30000, 160, 120, 16, 9),    # chunks of 256
    (1, 60000, 160, 120, 16, 9),    # 512 on 152 SMs
    (2, 90000, 160, 120, 16, 9),    # 1024
])
@pytest.mark.parametrize("full", [True, False])
def test_bin_scan_edges(case, full):
    torch_cuda()
    N = native()
    V, n, W, H, B, _ = case
    rec10, r = bin_case_records(case)
    cfg = N.make_config(W, H, B, 64, 0, rect_lists=True)
    ranges_o, vals_o = O.bin_lists(rec10[:, 0], rec10[:, 1], rec10[:, 9], r, V, n, W, H, B)
    cnt = len(vals_o)
    cap = cnt if full else cnt - 1
    vals, ranges, tord, ninst, st = gpu_bin(N, rec_to_gpu(rec10, r), n, V, cfg, cap)
    assert ninst == cnt and st == (0 if full else N.CGS_ERR_CAPACITY)
    rg, vv = gpu_lists(vals, ranges, cap)
    assert np.array_equal(rg, np.minimum(ranges_o, cap))
    if full:
        assert np.array_equal(vv, vals_o)
    to = tord.cpu().numpy()
    assert np.array_equal(np.sort(to), np.arange(len(rg)))
    lens = (ranges_o[:, 1].astype(np.int64) - ranges_o[:, 0])[to]
    assert np.all(np.diff(length_class(lens)) <= 0)
