"""The raster backward on both sides of the tile counts where it goes from four parts of a
tile in two list segments to whole lists, to two parts and to whole tiles (8, 16 and 32 tiles
per SM), against the oracle's."""
from __future__ import annotations

import numpy as np
import pytest

from gpu_util import field_grad_check, native, torch_cuda
from oracle import oracle as O
from synth import make_tiny_scene
from test_gpu_parity import (gpu_forward_from_rec, residual_sign_flags, round32, sg_from_gpu,
                             slots_in_flagged_tiles)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H,views", [(16, 16, 1), (33, 47, 3), (608, 512, 1), (609, 511, 1), (1024, 608, 1), (1023, 624, 1), (1216, 1023, 1),
                                       (1216, 1040, 1)])
@pytest.mark.parametrize("persistent", [True, False])
def test_raster_bwd_parts(W, H, views, persistent):
    torch = torch_cuda()
    N = native()
    n = 300
    sc = make_tiny_scene(seed=W + H, n=n, sh_degree=0, W=W, H=H, views=views, tile=16)
    pre = O.preprocess(sc.params, n, 0, sc.cams, W, H, 16)
    rec = round32(pre["rec"])
    ranges, vals = O.bin_records(rec, pre["radius"], views, n, W, H, 16)
    # targets off the render by at least 0.02: no residual's sign hangs on rounding
    bare = O.render_fwd(rec, ranges, vals, views, W, H, 16, sc.cams)
    rng = np.random.default_rng(W)
    off = lambda x: (x + rng.choice([-1.0, 1.0], x.shape) * rng.uniform(0.02, 0.1, x.shape)).astype(np.float32)  # noqa: E731
    tgt_rgb, tgt_d = off(bare["img"]), np.maximum(off(bare["depth"]), 0.0).astype(np.float32)
    fw = O.render_fwd(rec, ranges, vals, views, W, H, 16, sc.cams, (0.0, 0.0, 0.0), tgt_rgb, tgt_d, 0.1, tol=1e-5)
    out = gpu_forward_from_rec(N, sc, rec, pre, tgt_rgb, tgt_d, 64)
    sg = torch.zeros(views * n * 12, device="cuda")
    work = torch.full((1,), 7, dtype=torch.int32, device="cuda") if persistent else None
    N.cgs_raster_bwd(out["rec"], out["vals"], out["ranges"], out["order"], views, out["cfg"], out["w"], out["img"],
                     out["depth"], out["T"], out["last"], out["tr"], out["td"], out["dcount"], None, None, sg,
                     work=work)
    torch.cuda.synchronize()
    ref, mag = O.render_bwd(rec, ranges, vals, views, n, W, H, 16, sc.cams, fw["img"], fw["depth"], tgt_rgb, tgt_d,
                            fw["depth_count"], with_abs=True)
    flag = (fw["near"] != 0) | residual_sign_flags(fw["img"], tgt_rgb, fw["depth"], tgt_d)
    near = slots_in_flagged_tiles(flag, ranges, vals, W, H, 16, views * n)
    field_grad_check(sg_from_gpu(sg), ref, near, f"bwd parts {W}x{H}", mag=mag)
