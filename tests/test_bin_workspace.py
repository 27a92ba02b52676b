"""The binning workspace asked for once serves every smaller map of the same window."""
from __future__ import annotations

import pytest

from paper_2410_00486_gb300 import _native as N
from paper_2410_00486_gb300 import build as B


@pytest.mark.parametrize("V,W,H", [(1, 160, 120), (1, 1200, 680), (2, 640, 480), (3, 321, 247), (8, 640, 480)])
def test_workspace_grows_with_the_map(V, W, H):
    B.build()
    cfg = N.make_config(W, H)
    sizes = [N.cgs_bin_sort_workspace(1 << 20, n, V, cfg) for n in range(1, 400_000 // V, 173)]
    assert all(a <= b for a, b in zip(sizes, sizes[1:]))
