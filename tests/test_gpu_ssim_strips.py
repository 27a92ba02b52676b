"""The SSIM loss where a block walks several 32-row steps of its strip (large windows) and at
the strips' ends, against plain PyTorch in 64 bits."""
from __future__ import annotations

import pytest

from gpu_util import native, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H,V,steps", [(1203, 677, 4, 3), (1200, 672, 9, 8), (700, 1057, 5, 3), (2049, 31, 16, 8),
                                         (33, 33, 1, 1)])
def test_ssim_strips(W, H, V, steps):
    torch = torch_cuda()
    N = native()
    F = torch.nn.functional
    blocks = lambda k: -(-W // 32) * -(-(-(-H // 32)) // k) * 3 * V   # noqa: E731
    assert blocks(steps) >= 3000 or steps == 1
    assert steps == 8 or blocks(steps + 1) < 3000
    g = torch.Generator(device="cuda").manual_seed(W + H)
    low = torch.rand(V, 3, H // 9 + 2, W // 9 + 2, generator=g, device="cuda")
    img = F.interpolate(low, size=(H, W), mode="bilinear", align_corners=False).contiguous()
    tgt = (img + 0.05 * torch.randn(img.shape, generator=g, device="cuda")).contiguous()
    depth = torch.rand(V, H, W, generator=g, device="cuda") + 1
    tdepth = torch.where(torch.rand(V, H, W, generator=g, device="cuda") < 0.2, 0.0, depth + 0.1).contiguous()
    count = (tdepth > 0).sum((1, 2)).int()
    weight = torch.linspace(0.5, 2.0, V, device="cuda")
    cfg = N.make_config(W, H, lambda_depth=0.1)
    loss, dimg, dd = torch.zeros(V, device="cuda"), torch.empty_like(img), torch.empty_like(depth)
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    ws = torch.empty(N.cgs_ssim_workspace(V, cfg), dtype=torch.uint8, device="cuda")
    for _ in range(2):      # the second call starts from the first one's workspace
        N.cgs_ssim_loss(img, tgt, depth, tdepth, count, V, cfg, weight, 0.2, loss, dimg, dd, ws, st)
    k = torch.exp(-torch.arange(-5, 6, device="cuda", dtype=torch.float64) ** 2 / 4.5)
    k = k / k.sum()

    def blur(x):
        x = F.conv2d(x, k.reshape(1, 1, 1, 11), padding=(0, 5))
        return F.conv2d(x, k.reshape(1, 1, 11, 1), padding=(5, 0))

    for v in range(V):
        x = img[v].double().unsqueeze(1).requires_grad_(True)
        y = tgt[v].double().unsqueeze(1)
        mx, my = blur(x), blur(y)
        sx, sy, sxy = blur(x * x) - mx * mx, blur(y * y) - my * my, blur(x * y) - mx * my
        S = (2 * mx * my + 1e-4) * (2 * sxy + 9e-4) / ((mx * mx + my * my + 1e-4) * (sx + sy + 9e-4))
        res = (depth[v].double() - tdepth[v].double()).abs() * (tdepth[v] > 0)
        L = weight[v].double() * (0.8 * (x - y).abs().mean() + 0.2 * (1 - S.mean()) + 0.1 * res.sum() / count[v])
        gx = torch.autograd.grad(L, x)[0].squeeze(1)
        L = float(L.detach())
        assert abs(float(loss[v]) - L) <= 2e-5 * abs(L)
        err = (dimg[v].double() - gx)
        assert float(err.norm() / gx.norm()) < 1e-3 and float(err.abs().max() / gx.abs().max()) < 1e-3
        want = torch.where(tdepth[v] > 0, -0.1 * weight[v] / count[v], torch.zeros_like(depth[v]))
        torch.testing.assert_close(dd[v], want, rtol=1e-6, atol=0)
    assert int(st.item()) == 0
