"""The forward on both sides of the tile count (8 per SM) up to which a thread has one pixel:
the same images, bit for bit, as the work-counting forward's two pixels a thread, and the
oracle's."""
from __future__ import annotations

import numpy as np
import pytest

from gpu_util import PIX_TOL, native, round32, torch_cuda
from oracle import oracle as O
from synth import make_tiny_scene
from test_gpu_parity import gpu_forward_from_rec

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H,views", [(7, 5, 1), (33, 47, 3), (608, 512, 1), (609, 512, 1)])   # to 1216, 1248 tiles
@pytest.mark.parametrize("bd", [32, 256])
def test_render_fwd_one_pixel_a_thread(W, H, views, bd):
    torch = torch_cuda()
    N = native()
    n = 200
    sc = make_tiny_scene(seed=W, n=n, sh_degree=0, W=W, H=H, views=views, tile=16)
    pre = O.preprocess(sc.params, n, 0, sc.cams, W, H, 16)
    rec = round32(pre["rec"])
    ranges, vals = O.bin_records(rec, pre["radius"], views, n, W, H, 16)
    rng = np.random.default_rng(W)
    tgt_rgb = rng.uniform(0, 1, (views, 3, H, W)).astype(np.float32)
    tgt_d = rng.uniform(0, 3, (views, H, W)).astype(np.float32)
    fw = O.render_fwd(rec, ranges, vals, views, W, H, 16, sc.cams, (0.0, 0.0, 0.0), tgt_rgb, tgt_d, 0.1, tol=1e-5)
    out = gpu_forward_from_rec(N, sc, rec, pre, tgt_rgb, tgt_d, bd)
    ok = fw["near"] == 0
    assert np.abs(out["img"].cpu().numpy() - fw["img"]).max(1)[ok].max() < PIX_TOL
    np.testing.assert_allclose(out["loss"].cpu().numpy(), fw["loss_view"], rtol=1e-4)
    cfg = out["cfg"]
    cfg.count_work = 1
    img, depth, T = (torch.empty_like(out[k]) for k in ("img", "depth", "T"))
    last, loss, cnt = torch.empty_like(out["last"]), torch.empty_like(out["loss"]), torch.empty_like(out["dcount"])
    ws = torch.empty(N.cgs_render_fwd_workspace(views, cfg), dtype=torch.uint8, device="cuda")
    N.cgs_render_fwd(out["rec"], out["vals"], out["ranges"], out["order"], views, cfg, out["w"], out["tr"], out["td"],
                     img, depth, T, last, loss, cnt, ws)
    torch.cuda.synchronize()
    for a, b in ((img, "img"), (depth, "depth"), (T, "T"), (last, "last"), (cnt, "dcount")):
        assert torch.equal(a, out[b]), b
    torch.testing.assert_close(loss, out["loss"], rtol=1e-6, atol=0)
