"""Eq. 9's depth term where a strip's sum of residuals exceeds float32's range and the mean
does not: strips of one step and of the most (small views by the thousand)."""
from __future__ import annotations

import numpy as np
import pytest

from gpu_util import native, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V,W,H", [(1, 32, 32), (2, 45, 256), (1000, 32, 256)])
def test_depth_term_of_large_residuals(V, W, H):
    torch = torch_cuda()
    N = native()
    cfg = N.make_config(W, H)
    g = torch.Generator(device="cuda").manual_seed(V)
    img = torch.rand(V, 3, H, W, device="cuda", generator=g)
    depth, big = torch.zeros(V, H, W, device="cuda"), np.float32(1e36)
    tgt = torch.full_like(depth, float(big))
    count = torch.full((V,), H * W, dtype=torch.int32, device="cuda")
    loss, dimg, dd = torch.zeros(V, device="cuda"), torch.empty_like(img), torch.empty_like(depth)
    ws = torch.empty(N.cgs_ssim_workspace(V, cfg), dtype=torch.uint8, device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    N.cgs_ssim_loss(img, img, depth, tgt, count, V, cfg, None, 0.2, loss, dimg, dd, ws, st)
    assert int(st.item()) == 0
    # equal images: the depth term alone; a thread's four residuals and the result are rounded
    want = float(np.float32(0.1)) * float(big)
    np.testing.assert_allclose(loss.cpu().numpy(), want, rtol=6 * 2.0 ** -24)
    assert torch.equal(dd, torch.full_like(dd, -float(np.float32(0.1) / np.float32(H * W))))
