"""The fused loss where a view's sum of residuals exceeds float32's range though its mean does
not, on windows of one and of several blocks' tiles: the sums are kept in double."""
from __future__ import annotations

import numpy as np
import pytest

from gpu_util import native, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H,V", [(160, 120, 1), (512, 256, 1), (528, 256, 3), (1199, 677, 2), (4096, 512, 1)])
def test_loss_of_large_residuals(W, H, V):
    torch = torch_cuda()
    N = native()
    cfg = N.make_config(W, H, 16, 64, 0)
    tiles = N.cgs_tiles_per_view(cfg) * V
    z = lambda *s, dtype=torch.float32: torch.zeros(s, dtype=dtype, device="cuda")   # noqa: E731
    # no splats: the image is the black background, every residual the target itself
    rgb, depth, big = z(V, 3, H, W), z(V, H, W), np.float32(1e35)
    rgb[:] = float(big)
    depth[:, ::2] = float(big)          # the other rows have no valid depth
    img, d, T = z(V, 3, H, W), z(V, H, W), z(V, H, W)
    last, loss, count = z(V, H, W, dtype=torch.int32), z(V), z(V, dtype=torch.int32)
    weight = torch.arange(1, V + 1, dtype=torch.float32, device="cuda")
    ws = torch.empty(N.cgs_render_fwd_workspace(V, cfg), dtype=torch.uint8, device="cuda")
    st = z(1, dtype=torch.int32)
    N.cgs_render_fwd(z(12), z(1, dtype=torch.int32), z(2 * tiles, dtype=torch.int32), None, V, cfg, weight, rgb, depth,
                     img, d, T, last, loss, count, ws, st)
    assert int(st.item()) == 0
    assert count.tolist() == [W * ((H + 1) // 2)] * V
    # a tile's sums are float32: at most 14 roundings (pixels, warps and blocks of a tile) of 2^-24
    want = np.arange(1, V + 1) * float(big) * 1.1
    np.testing.assert_allclose(loss.cpu().numpy(), want, rtol=14 * 2.0 ** -24)
