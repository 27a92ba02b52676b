"""Point clouds with coordinates that are not finite: the status says so, and the finite
points' scales come from the finite points alone, or take the floor where too few are left."""
from __future__ import annotations

import numpy as np
import pytest

from gpu_util import native, torch_cuda
from oracle import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,bad,value", [(4, 1, np.nan), (4, 1, np.inf), (4, 3, -np.inf), (3, 1, np.nan), (2, 1, np.nan),
                                         (5, 1, np.nan), (5, 1, np.inf), (300, 40, np.nan), (5000, 7, -np.inf),
                                         (6, 6, np.nan)])
def test_nonfinite_points(m, bad, value):
    torch = torch_cuda()
    N = native()
    rng = np.random.default_rng(m + bad)
    xyz = rng.normal(size=(m, 3)).astype(np.float32)
    rows = rng.choice(m, bad, replace=False)
    xyz[rows, rng.integers(0, 3, bad)] = value
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()   # noqa: E731
    out = [torch.full((N.cgs_param_count(m, 0),), 7.0, device="cuda") for _ in range(3)]
    ws = torch.full((N.cgs_points_workspace(m),), 0xff, dtype=torch.uint8, device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    N.cgs_points_to_gaussians(None, None, None, 0, 0, t(xyz), t(np.full_like(xyz, 0.5)), m, 0.1, ws, *out, st)
    assert int(st.item()) == N.CGS_ERR_NONFINITE
    good = np.isfinite(xyz).all(1)
    logs = out[0][3 * m: 6 * m].reshape(m, 3).cpu().numpy()[good]
    want, k = int(good.sum()) - 1, min(3, m - 1)
    d2 = np.zeros(good.sum()) if want < k else O.knn_mean_d2(xyz[good])
    # as for finite clouds: a mean of float32 distances and its logarithm
    np.testing.assert_allclose(logs, np.repeat(0.5 * np.log(np.maximum(d2, 1e-7))[:, None], 3, 1), rtol=0, atol=2e-6)
