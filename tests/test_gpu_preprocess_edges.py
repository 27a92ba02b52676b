"""The projection's backward at the edges of its blocks of 128 Gaussians, of its chunks of 32
views and of its 16-byte copies, against the oracle's chain rule on the same slot gradients."""
from __future__ import annotations

import numpy as np
import pytest

from gpu_util import native, param_grad_check, torch_cuda
from oracle import oracle as O
from synth import make_tiny_scene
from test_gpu_parity import cfg_for, gaussians_of_slots, gpu_scene_tensors, round32, sg_to_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,views,deg", [(1, 1, 0), (127, 1, 3), (128, 33, 1), (130, 31, 2), (257, 32, 3), (96, 70, 3)])
def test_preprocess_bwd_edges(n, views, deg):
    torch = torch_cuda()
    N = native()
    sc = make_tiny_scene(seed=n + views, n=n, sh_degree=deg, W=64, H=48, views=views, tile=16)
    pre = O.preprocess(sc.params, n, deg, sc.cams, sc.width, sc.height, sc.tile)
    rng = np.random.default_rng(n)
    keep = (pre["radius"] > 0) & (pre["fragile"] == 0)
    sg = round32(rng.normal(0, 1e-3, (views * n, 10)) * keep[:, None])
    params, cams = gpu_scene_tensors(sc)
    cfg = cfg_for(N, sc)
    rec = torch.zeros(views * n * 12, device="cuda")
    N.cgs_preprocess(params, n, cams, views, cfg, rec, None)
    start = torch.randn(params.numel(), device="cuda")
    grads, added = torch.full_like(start, float("nan")), start.clone()
    acc, den, mx = (torch.zeros(n, device="cuda") for _ in range(3))
    N.cgs_preprocess_bwd(params, n, cams, views, cfg, rec, sg_to_gpu(sg), grads, False, acc, den, mx)
    N.cgs_preprocess_bwd(params, n, cams, views, cfg, rec, sg_to_gpu(sg), added, True)
    torch.cuda.synchronize()
    assert torch.equal(added, start + grads)
    ref = O.preprocess_bwd(sc.params, n, deg, sc.cams, sc.width, sc.height, sc.tile, sg)
    param_grad_check(grads.cpu().numpy().astype(np.float64), ref, n, deg, gaussians_of_slots(pre["fragile"] > 0, n),
                     f"pre bwd n={n} V={views}", l2=1e-4)
    a_o, d_o, m_o = O.densify_stats(sg, pre["radius"], views, n, sc.width, sc.height)
    np.testing.assert_allclose(acc.cpu().numpy(), a_o, rtol=1e-5, atol=1e-9)
    solid = ~gaussians_of_slots(pre["fragile"] > 0, n)
    assert np.array_equal(den.cpu().numpy()[solid], d_o[solid])
    assert np.array_equal(mx.cpu().numpy()[solid], m_o[solid])
