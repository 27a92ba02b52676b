"""Densification and point insertion at the sizes where their kernels change course: block
and span edges, blocks of one kind of Gaussian, a caller's n_out below the plan's, and clouds
whose points need the whole-grid search."""
from __future__ import annotations

import numpy as np
import pytest

from gpu_util import native, torch_cuda
from oracle import oracle as O
from test_gpu_parity import _check_new_gaussians, _gpu_points

pytestmark = pytest.mark.gpu


def _plan(n, deg, codes, seed):
    """A map whose Gaussian g gets code codes[g] (0 prune, 1 keep, 2 clone, 3 split)."""
    rng = np.random.default_rng(seed)
    P = rng.normal(size=(14 + 3 * ((deg + 1) ** 2 - 1)) * n).astype(np.float32)
    P[3 * n: 6 * n] = np.repeat(np.where(codes == 3, -1.0, -6.0), 3).astype(np.float32)
    P[10 * n: 11 * n] = np.where(codes == 0, -9.0, 0.5).astype(np.float32)
    return P, np.where(codes >= 2, 1.0, 0.0).astype(np.float32), np.ones(n, np.float32)


@pytest.mark.parametrize("n,deg,kind", [(1, 0, "split"), (127, 1, "mix"), (128, 2, "clone"), (129, 3, "mix"),
                                        (1025, 3, "split"),
                                        (3000, 0, "prune-blocks")])
@pytest.mark.parametrize("short", [0, 3])
def test_densify_edges(n, deg, kind, short):
    torch = torch_cuda()
    N = native()
    rng = np.random.default_rng(n + deg)
    codes = {"split": np.full(n, 3), "clone": np.full(n, 2)}.get(kind, rng.integers(0, 4, n))
    if kind == "prune-blocks":
        codes[128:640] = 0
    P, accum, denom = _plan(n, deg, codes, n)
    M, V = rng.normal(size=P.size).astype(np.float32), rng.uniform(size=P.size).astype(np.float32)
    normals = rng.normal(size=(n, 2, 3)).astype(np.float32)
    code_o, _ = O.densify_plan(P, n, deg, accum, denom, 0.5, 0.01, 0.02)
    np.testing.assert_array_equal(code_o, codes)
    P_o, M_o, V_o, n_o = O.densify_apply(P, M, V, n, deg, code_o, normals)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()   # noqa: E731
    ws = torch.empty(N.cgs_densify_workspace(n), dtype=torch.uint8, device="cuda")
    nout = torch.zeros(1, dtype=torch.int64, device="cuda")
    N.cgs_densify_plan(t(P), n, deg, t(accum), t(denom), 0.5, 0.01, 0.02, ws, nout)
    assert int(nout.item()) == n_o
    room = max(1, n_o - short)       # below the plan's count the last Gaussians are left out
    size = N.cgs_param_count(room, deg)
    out = [torch.full((size + 64,), 7.0, device="cuda") for _ in range(3)]
    N.cgs_densify_apply(t(P), t(M), t(V), n, deg, ws, t(normals), room, *out)
    torch.cuda.synchronize()
    # a split child's mean R(q) (s z): |s z| < 3.2 here, R's entries and the sums good to about
    # 12 half-ulps of it
    widths = [3, 3, 4, 1, 3, 3 * ((deg + 1) ** 2 - 1)]
    whole = room if room >= n_o else room - 1     # the last kept output may be half a pair
    for got, want, tol in zip(out, (P_o, M_o, V_o), (2e-6, 0, 0)):
        got = got.cpu().numpy()
        assert np.all(got[size:] == 7.0)
        oi = oo = 0
        for w in widths:
            np.testing.assert_allclose(got[oo: oo + w * whole], want[oi: oi + w * whole].astype(np.float32), rtol=tol,
                                       atol=5e-6 if tol else 0)
            oi += w * n_o
            oo += w * room


def test_densify_more_than_one_chunk_per_span():
    """2^20 + 1 Gaussians: each block of the scan walks several chunks."""
    torch = torch_cuda()
    N = native()
    n, deg = (1 << 20) + 1, 0
    rng = np.random.default_rng(5)
    codes = rng.integers(0, 2, n)
    P, accum, denom = _plan(n, deg, codes, 6)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()   # noqa: E731
    ws = torch.empty(N.cgs_densify_workspace(n), dtype=torch.uint8, device="cuda")
    nout = torch.zeros(1, dtype=torch.int64, device="cuda")
    p, z = t(P), torch.zeros(P.size, device="cuda")
    N.cgs_densify_plan(p, n, deg, t(accum), t(denom), 0.5, 0.01, 0.02, ws, nout)
    n_out = int(nout.item())
    assert n_out == int(codes.sum())
    out = [torch.empty(N.cgs_param_count(n_out, deg), device="cuda") for _ in range(3)]
    N.cgs_densify_apply(p, p, z, n, deg, ws, torch.zeros(n, 2, 3, device="cuda"), n_out, *out)
    keep = t(codes.astype(bool))
    want = torch.cat([x.reshape(n, -1)[keep].reshape(-1) for x in p.split([3 * n, 3 * n, 4 * n, n, 3 * n])])
    assert torch.equal(out[0], want) and torch.equal(out[1], want) and not out[2].any()


@pytest.mark.parametrize("m,far", [(5, 1), (127, 20), (700, 300), (4097, 40), (20000, 6)])
def test_points_far_from_the_others(m, far):
    """A dense cluster with some points far apart from it and from each other."""
    N = native()
    rng = np.random.default_rng(m)
    xyz = rng.normal(0, 0.05, (m, 3))
    xyz[rng.choice(m, far, replace=False)] = rng.uniform(-30, 30, (far, 3))
    xyz = xyz.astype(np.float32)
    rgb = rng.uniform(0, 1, xyz.shape).astype(np.float32)
    got, _, _ = _gpu_points(N, xyz, rgb, 1)
    _check_new_gaussians(got, xyz, rgb, 1, 0, O.knn_mean_d2(xyz))
