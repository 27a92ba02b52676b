"""The binning workspace of a larger map covers every smaller one, also where the map's size
changes the chunks that the sort takes (256 to 2048 slots, by blocks per multiprocessor)."""
from __future__ import annotations

import pytest

from paper_2410_00486_gb300 import _native as N
from paper_2410_00486_gb300 import build as B


@pytest.mark.parametrize("V,W,H", [(1, 1200, 680), (3, 637, 479), (8, 640, 480), (12, 640, 480), (16, 1200, 680),
                                   (700, 64, 48)])
def test_workspace_covers_smaller_maps(V, W, H):
    B.build()
    cfg = N.make_config(W, H)
    # every chunk size's edges, beyond the largest step for up to 200 multiprocessors
    last = max(4096, 2 * 4 * 200 * 2048 // V)
    edges = {e + d for e in range(0, last, 256) for d in (0, 1, 2)} - {0}
    sizes = [N.cgs_bin_sort_workspace(1 << 20, n, V, cfg) for n in sorted(edges)]
    assert all(a <= b for a, b in zip(sizes, sizes[1:]))
