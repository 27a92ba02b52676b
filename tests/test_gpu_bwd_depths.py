"""The raster backward's batch depths on a window of whole tiles (more than 32 tiles per SM),
where every depth is a kernel of its own, against the oracle's."""
from __future__ import annotations

import numpy as np
import pytest

from gpu_util import field_grad_check, native, torch_cuda
from oracle import oracle as O
from synth import make_tiny_scene
from test_gpu_parity import (gpu_forward_from_rec, residual_sign_flags, round32, sg_from_gpu,
                             slots_in_flagged_tiles)

pytestmark = pytest.mark.gpu

W, H, N_GAUSS = 1232, 1040, 3000       # 77 x 65 = 5005 tiles for 152 SMs, lists of several hundred faint splats


@pytest.fixture(scope="module")
def window():
    sc = make_tiny_scene(seed=9, n=N_GAUSS, sh_degree=0, W=W, H=H, views=1, tile=16,
                         opacity_mean=-3.0)
    pre = O.preprocess(sc.params, N_GAUSS, 0, sc.cams, W, H, 16)
    rec = round32(pre["rec"])
    ranges, vals = O.bin_records(rec, pre["radius"], 1, N_GAUSS, W, H, 16)
    # targets off the render by at least 0.02: no residual's sign hangs on rounding
    bare = O.render_fwd(rec, ranges, vals, 1, W, H, 16, sc.cams)
    rng = np.random.default_rng(W)
    off = lambda x: (x + rng.choice([-1.0, 1.0], x.shape) * rng.uniform(0.02, 0.1, x.shape)).astype(np.float32)  # noqa: E731
    tgt_rgb, tgt_d = off(bare["img"]), np.maximum(off(bare["depth"]), 0.0).astype(np.float32)
    fw = O.render_fwd(rec, ranges, vals, 1, W, H, 16, sc.cams, (0.0, 0.0, 0.0), tgt_rgb, tgt_d, 0.1, tol=1e-5)
    ref, mag = O.render_bwd(rec, ranges, vals, 1, N_GAUSS, W, H, 16, sc.cams, fw["img"], fw["depth"], tgt_rgb, tgt_d,
                            fw["depth_count"], with_abs=True)
    flag = (fw["near"] != 0) | residual_sign_flags(fw["img"], tgt_rgb, fw["depth"], tgt_d)
    return sc, pre, rec, tgt_rgb, tgt_d, ref, mag, slots_in_flagged_tiles(flag, ranges, vals, W, H, 16, N_GAUSS)


@pytest.mark.parametrize("depth", [32, 64, 128, 256])
@pytest.mark.parametrize("persistent", [True, False])
def test_raster_bwd_depths(window, depth, persistent):
    torch = torch_cuda()
    N = native()
    sc, pre, rec, tgt_rgb, tgt_d, ref, mag, near = window
    cfg = N.make_config(W, H, 16, 64, 0, batch_depth_bwd=depth)
    assert N.cgs_raster_bwd_batch(1, cfg) == depth
    out = gpu_forward_from_rec(N, sc, rec, pre, tgt_rgb, tgt_d, 64)
    assert int(out["last"].max()) > 256          # more than one batch of every depth
    sg = torch.zeros(N_GAUSS * 12, device="cuda")
    work = torch.full((1,), 7, dtype=torch.int32, device="cuda") if persistent else None
    N.cgs_raster_bwd(out["rec"], out["vals"], out["ranges"], out["order"], 1, cfg, out["w"], out["img"], out["depth"],
                     out["T"], out["last"], out["tr"], out["td"], out["dcount"], None, None, sg, work=work)
    torch.cuda.synchronize()
    field_grad_check(sg_from_gpu(sg), ref, near, f"bwd depth {depth}", mag=mag)
