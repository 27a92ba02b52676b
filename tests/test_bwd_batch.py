"""The batch depth that the raster backward takes, and the autotuner's candidates: a depth
that a window of few tiles does not take is measured no second time."""
from __future__ import annotations

import pytest
import torch

from paper_2410_00486_gb300 import _native as N
from paper_2410_00486_gb300 import autotune as A
from paper_2410_00486_gb300 import build as B


@pytest.mark.parametrize("tile,W,H,V,fixed", [(16, 16, 16, 1, True), (16, 1200, 680, 1, True), (16, 1200, 680, 16, False),
                                              (8, 160, 120, 1, False), (32, 160, 120, 1, False)])
def test_depth_taken(tile, W, H, V, fixed):
    B.build()
    for d in (32, 64, 128, 256):
        assert N.cgs_raster_bwd_batch(V, N.make_config(W, H, tile, d)) == (32 if fixed else d)
        assert N.cgs_raster_bwd_batch(V, N.make_config(W, H, tile, 128, batch_depth_bwd=d)) == (32 if fixed else d)
    assert N.cgs_raster_bwd_batch(0, N.make_config(W, H, tile)) == N.CGS_ERR_ARG


@pytest.mark.parametrize("tile,W,H,V,windows", [(16, 640, 480, 1, 4), (16, 1200, 680, 16, 4 + 3 + 3),
                                                (8, 640, 480, 1, 4 + 3 + 3)])
def test_autotuner_measures_each_shape_once(monkeypatch, tile, W, H, V, windows):
    B.build()
    built = []

    class Window:
        def __init__(self, params, n, deg, width, height, views, tile, batch_depth, batch_depth_bwd):
            built.append((tile, batch_depth, N.cgs_raster_bwd_batch(views, N.make_config(
                width, height, tile, batch_depth, batch_depth_bwd=batch_depth_bwd))))

        def set_window(self, *a):
            pass

        def fit_capacity(self, *a):
            pass

        def read_status(self):
            return 0, 0

    monkeypatch.setattr(A, "MappingWindow", Window)
    monkeypatch.setattr(A, "time_window", lambda win, reps: 1.0 + len(built))
    A._memo.clear()
    best, ms = A.autotune(torch.zeros(1), 1, 0, W, H, torch.zeros(V, 20), None, None,
                          candidates=[(tile, d) for d in (32, 64, 128, 256)])
    A._memo.clear()
    assert len(built) == len(set(built)) == len(ms) == windows
    assert best == built[0]              # the fake's times grow from window to window
