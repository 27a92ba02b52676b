"""A cloud with several hundred points too far apart for the near search (621 on this cloud,
for 304 blocks of the whole-grid search), so that blocks take more than one of them."""
from __future__ import annotations

import numpy as np
import pytest

from gpu_util import native
from oracle import oracle as O
from test_gpu_parity import _check_new_gaussians, _gpu_points

pytestmark = pytest.mark.gpu


def test_more_far_points_than_blocks():
    N = native()
    m, far = 20000, 900
    rng = np.random.default_rng(m)
    xyz = rng.normal(0, 3, (m, 3))
    xyz[rng.choice(m, far, replace=False)] = rng.uniform(-30, 30, (far, 3))
    xyz = xyz.astype(np.float32)
    rgb = rng.uniform(0, 1, xyz.shape).astype(np.float32)
    got, _, _ = _gpu_points(N, xyz, rgb, 0)
    _check_new_gaussians(got, xyz, rgb, 0, 0, O.knn_mean_d2(xyz))
