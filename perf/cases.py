"""Performance cases of the mapping library: the work a mapping program has it do, through
its public entry points (`MappingWindow`, the autograd functions, the C-ABI binding).

A case is a dict of plain values; `op` says which entry point it goes through:

  iter      MappingWindow.forward + backward: render a window of keyframes, its loss, and the
            gradients and densification statistics (captured into a CUDA graph where `graph`
            is set, as a program does for windows whose launches would otherwise show)
  autograd  RenderWindow under a loss the caller wrote in torch
  render    MappingWindow.forward without a loss: views for evaluation or display
  ssim      cgs_ssim_loss: the photometric loss of Eq. 9 and its pixel gradients
  adam      MappingWindow.optimizer_step
  densify   cgs_densify_plan + cgs_densify_apply: clone, split and prune
  points    cgs_points_to_gaussians: a new keyframe's point cloud becomes Gaussians

Scenes are the repository's synthetic ones (box and room), drawn on the GPU from the seed;
keyframe images are smooth random RGB-D frames with an invalid depth band, so inputs depend
on nothing but the seed.
"""
from __future__ import annotations

import math

import torch

from paper_2410_00486_gb300 import _native as N
from paper_2410_00486_gb300.autograd import RenderWindow
from paper_2410_00486_gb300.window import MappingWindow

Y00 = 0.28209479177387814
BG = (0.1, 0.2, 0.3)
LAMBDA_DEPTH = 0.1
LR = (1.6e-4, 5e-3, 1e-3, 2.5e-2, 2.5e-3, 2.5e-3 / 20.0)
BETAS, EPS, LAMBDA_O = (0.9, 0.999), 1e-15, 0.01
TAU_P, SCALE_THR, EPS_ALPHA = 0.001, 0.03, 0.02
INIT_OPACITY = 0.1


def _iter(name, scene, n, deg, w, h, views, *, depths=(64, 0), graph=False, ssim=0.0, opac=(0.0, 1.0), op="iter"):
    c = dict(op=op, scene=scene, n=n, sh_degree=deg, width=w, height=h, views=views, batch_depth=depths[0],
             batch_depth_bwd=depths[1], graph=graph, lambda_ssim=ssim, opacity_mean=opac[0], opacity_std=opac[1])
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest mapping iteration: a few thousand Gaussians in one small image, where
        # launches and latency are all there is
        _iter("view_2k_sh0_160x120", "box", 2000, 0, 160, 120, 1, graph=True),
        # a caller's own loss through torch.autograd on a small view, launched call by call
        _iter("autograd_5k_sh1_320x240", "box", 5000, 1, 320, 240, 1, op="autograd"),
        # one keyframe of a TUM-sized map at the Gaussian count the paper reports for it: the
        # ordinary call of the sequential mapping loop
        _iter("view_40k_sh3_640x480", "room", 40_000, 3, 640, 480, 1, graph=True),
        # one keyframe of a Replica-sized map
        _iter("view_100k_sh3_1200x680", "room", 100_000, 3, 1200, 680, 1, depths=(128, 32), graph=True),
        # a keyframe window with very uneven visibility (150k to 20k of 200k Gaussians)
        _iter("window8_200k_sh3_640x480", "path", 200_000, 3, 640, 480, 8, depths=(128, 32)),
        # the largest window: long per-pixel lists from many faint Gaussians
        _iter("window16_300k_sh3_1200x680", "room", 300_000, 3, 1200, 680, 16, depths=(128, 32), opac=(-1.0, 1.5)),
        # a small window with the paper's whole loss (Eq. 9), odd image sizes and counts
        _iter("window3_ssim_60k_sh2_637x479", "room", 60_001, 2, 637, 479, 3, ssim=0.2),
        # four views rendered for evaluation, no loss and no gradients, ragged tiles
        _iter("render4_90k_sh3_1199x677", "room", 90_001, 3, 1199, 677, 4, op="render"),
        # the loss of Eq. 9 on its own, as a program with its own renderer loop calls it
        dict(name="ssim_4x1200x680", op="ssim", width=1200, height=680, views=4, lambda_ssim=0.2),
        # one optimiser step on the largest map
        dict(name="adam_300k_sh3", op="adam", n=300_000, sh_degree=3),
        # density control of a grown map, every few hundred iterations
        dict(name="densify_200k_sh3", op="densify", n=200_000, sh_degree=3),
        # a 640x480 depth frame's points join a map of 100k Gaussians
        dict(name="points_307k_onto_100k_sh3", op="points", n=100_000, sh_degree=3, points=307_200),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    op = rng.choice(["iter", "iter", "iter", "iter", "autograd", "render", "ssim", "adam", "densify", "points"])
    if op == "adam" or op == "densify":
        return dict(op=op, n=int(_log_uniform(rng, 5e3, 3e5)), sh_degree=rng.choice([0, 1, 2, 3, 3]))
    if op == "points":
        return dict(op=op, n=int(_log_uniform(rng, 2e3, 1e5)), sh_degree=rng.choice([0, 1, 2, 3, 3]),
                    points=int(_log_uniform(rng, 2e3, 3e5)))
    w = int(_log_uniform(rng, 160, 1200))
    h = max(97, int(w * rng.uniform(0.55, 0.8)))
    if op == "ssim":
        return dict(op=op, width=w, height=h, views=rng.randint(1, 8), lambda_ssim=rng.choice([0.2, 0.2, 0.5]))
    # Gaussians per pixel as in the repository's workloads (0.065 to 0.65)
    n = min(250_000, max(2000, int(w * h * _log_uniform(rng, 0.065, 0.65))))
    views = rng.choice([1, 1, 2, 3, 5, 8, 12]) if op == "iter" else rng.choice([1, 1, 2, 4])
    scene = rng.choice(["room", "room", "path"]) if n > 8000 else "box"
    return _iter(None, scene, n, rng.choice([0, 1, 2, 3, 3]), w, h, views,
                 depths=rng.choice([(64, 0), (128, 32)]), graph=op == "iter" and views <= 2,
                 ssim=0.2 if op == "iter" and rng.random() < 0.25 else 0.0,
                 opac=rng.choice([(0.0, 1.0), (-1.0, 1.5)]), op=op)


# ------------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _rand(g, lo, hi, *size):
    return lo + (hi - lo) * torch.rand(*size, generator=g, device="cuda")


def _normal(g, mean, std, *size):
    return mean + std * torch.randn(*size, generator=g, device="cuda")


def _room_points(g, n):
    """70% on the floor and four walls of a 6x5x3 m room (by area, 2 cm jitter), 30% inside."""
    a, b = _rand(g, 0, 1, n), _rand(g, 0, 1, n)
    jit = _normal(g, 0.0, 0.02, n)
    which = torch.searchsorted(torch.tensor([30.0, 45.0, 60.0, 78.0], device="cuda"), _rand(g, 0, 96, n))
    inside = _rand(g, 0, 1, n) < 0.3
    x, y, z = -3 + 6 * a, 3 * b, -2.5 + 5 * b
    p = torch.stack([x, jit, z], 1)                                           # floor
    p = torch.where((which == 1)[:, None], torch.stack([-3 + jit, 3 * a, z], 1), p)
    p = torch.where((which == 2)[:, None], torch.stack([3 + jit, 3 * a, z], 1), p)
    p = torch.where((which == 3)[:, None], torch.stack([x, y, -2.5 + jit], 1), p)
    p = torch.where((which == 4)[:, None], torch.stack([x, y, 2.5 + jit], 1), p)
    free = torch.stack([_rand(g, -3, 3, n), _rand(g, 0, 3, n), _rand(g, -2.5, 2.5, n)], 1)
    return torch.where(inside[:, None], free, p)


def _params(g, scene, n, deg, opac_mean=0.0, opac_std=1.0):
    if scene == "box":
        means = torch.stack([_rand(g, -2, 2, n), _rand(g, -1.5, 1.5, n), _rand(g, 1, 4, n)], 1)
    else:
        means = _room_points(g, n)
    q = _normal(g, 0.0, 1.0, n, 4)
    k = (deg + 1) ** 2
    parts = [means, _normal(g, -3.5, 0.5, n, 3), q / q.norm(dim=1, keepdim=True), _normal(g, opac_mean, opac_std, n),
             _normal(g, 0.0, 0.2 / Y00, n, 3), _normal(g, 0.0, 0.05, n, k - 1, 3)]
    return torch.cat([p.reshape(-1) for p in parts]).float()


def _cross(a, b):
    return [a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]]


def _unit(a):
    s = math.sqrt(sum(x * x for x in a))
    return [x / s for x in a]


def _cams(scene, views, w, h):
    """Pinhole cameras float32 [V, 20]: identity (box), on an ellipse in the room looking at
    its centre (room), or on a straight path along the room whose yaw turns away (path)."""
    rows = []
    f = {"box": 0.9375 * w, "room": 0.5 * w, "path": 0.82 * w}[scene]
    for i in range(views):
        if scene == "box":
            R, t = [[1, 0, 0], [0, 1, 0], [0, 0, 1]], [0.02 * i, 0, 0]
        else:
            if scene == "room":
                th = 2 * math.pi * i / views
                pos = [2.0 * math.cos(th), 1.4, 1.5 * math.sin(th)]
                fwd = [-pos[0], 1.5 - pos[1], -pos[2]]
            else:
                a = i / max(views - 1, 1)
                pos, yaw = [0.0, 1.6, -4.85 + 2.0 * a], 1.5 * a
                fwd = [math.sin(yaw), -0.15, math.cos(yaw)]
            fwd = _unit(fwd)
            right = _unit(_cross([0.0, -1.0, 0.0], fwd))
            R = [right, _cross(fwd, right), fwd]
            t = [-sum(r[k] * pos[k] for k in range(3)) for r in R]
        rows.append([x for r in R for x in r] + list(t) + [f, f, w / 2 - 0.5, h / 2 - 0.5, 1.0, 0.0, 0.0, 0.0])
    return torch.tensor(rows, dtype=torch.float32, device="cuda")


def _frames(g, views, w, h):
    """Smooth RGB frames with fine texture, and depth with an invalid band."""
    low = _rand(g, 0, 1, views, 4, max(2, h // 40), max(2, w // 40))
    x = torch.nn.functional.interpolate(low, size=(h, w), mode="bilinear", align_corners=False)
    rgb = (x[:, :3] + _normal(g, 0.0, 0.03, views, 3, h, w)).clamp(0, 1).contiguous()
    depth = (0.5 + 4.5 * x[:, 3] + _normal(g, 0.0, 0.02, views, h, w)).contiguous()
    depth[:, : max(1, h // 8)] = 0.0
    return rgb, depth


def _weights(views):
    return torch.tensor([1.0 + (i % 3 == 2) for i in range(views)], device="cuda")   # scheduler multiplicities


def _window_inputs(case, seed):
    g = _gen(seed)
    p = _params(g, case["scene"], case["n"], case["sh_degree"], case["opacity_mean"], case["opacity_std"])
    cams = _cams(case["scene"], case["views"], case["width"], case["height"])
    rgb, depth = _frames(g, case["views"], case["width"], case["height"])
    return p, cams, rgb, depth, _weights(case["views"])


def _adam_inputs(case, seed):
    g = _gen(seed)
    p = _params(g, "room", case["n"], case["sh_degree"])
    unseen = _rand(g, 0, 1, p.numel()) < 0.2          # out of every view: zero gradient, old moments
    grad = torch.where(unseen, torch.zeros_like(p), _normal(g, 0.0, 1e-5, p.numel()))
    return p, grad, _normal(g, 0.0, 1e-6, p.numel()), _normal(g, 0.0, 1e-6, p.numel()).square()


def _densify_inputs(case, seed):
    g = _gen(seed)
    n = case["n"]
    p = _params(g, "room", n, case["sh_degree"], 0.0, 2.0)
    m, v = _normal(g, 0.0, 1e-5, p.numel()), _normal(g, 0.0, 1e-5, p.numel()).square()
    denom = torch.randint(0, 200, (n,), generator=g, device="cuda").float()
    accum = denom * torch.exp(_normal(g, math.log(4e-4), 1.0, n))
    return p, m, v, accum, denom, _normal(g, 0.0, 1.0, n, 2, 3)


def _points_inputs(case, seed):
    g = _gen(seed)
    p = _params(g, "room", case["n"], case["sh_degree"])
    m, v = _normal(g, 0.0, 1e-5, p.numel()), _normal(g, 0.0, 1e-5, p.numel()).square()
    k = case["points"]
    xyz = _room_points(g, k)
    rep = max(1, k // 100)                           # quantised depth repeats points exactly
    xyz[2:2 + rep] = xyz[torch.randint(2 + rep, k, (rep,), generator=g, device="cuda")]
    xyz[:2] = _rand(g, -40, 40, 2, 3)                # stray measurements far outside
    xyz = xyz[torch.randperm(k, generator=g, device="cuda")].contiguous()
    return p, m, v, xyz, _rand(g, 0, 1, k, 3)


def prepare(case, seed):
    s = dict(case=case)
    op = case["op"]
    if op in ("iter", "autograd", "render"):
        p, cams, rgb, depth, weight = _window_inputs(case, seed)
        win = MappingWindow(p, case["n"], case["sh_degree"], case["width"], case["height"], case["views"], tile=16,
                            batch_depth=case["batch_depth"], batch_depth_bwd=case["batch_depth_bwd"],
                            lambda_depth=LAMBDA_DEPTH, bg=BG, lambda_ssim=case["lambda_ssim"])
        win.set_window(cams, rgb, depth, weight)
        win.fit_capacity()
        s.update(win=win)
        if op == "autograd":
            s.update(params=p.clone().requires_grad_(True), rgb=rgb, depth=depth, valid=depth > 0)
        if case["graph"]:
            s.update(graph=torch.cuda.CUDAGraph())
            torch.cuda.synchronize()
            with torch.cuda.graph(s["graph"]):
                win.forward()
                win.backward()
    elif op == "ssim":
        g = _gen(seed)
        V, w, h = case["views"], case["width"], case["height"]
        rgb, depth = _frames(g, V, w, h)
        img = (rgb + _normal(g, 0.0, 0.05, V, 3, h, w)).contiguous()
        rendered = (depth + _normal(g, 0.0, 0.05, V, h, w)).contiguous()
        cfg = N.make_config(w, h, lambda_depth=LAMBDA_DEPTH)
        s.update(rgb=rgb, depth=depth, img=img, rendered=rendered, cfg=cfg, weight=_weights(V),
                 count=(depth > 0).sum((1, 2)).int(), loss=torch.zeros(V, device="cuda"),
                 dimg=torch.empty_like(img), ddepth=torch.empty_like(depth),
                 status=torch.zeros(1, dtype=torch.int32, device="cuda"),
                 ws=torch.empty(N.cgs_ssim_workspace(V, cfg), dtype=torch.uint8, device="cuda"))
    elif op == "adam":
        p, grad, m, v = _adam_inputs(case, seed)
        win = MappingWindow(p, case["n"], case["sh_degree"], 64, 48, 1, lr=LR, betas=BETAS, eps=EPS,
                            lambda_o=LAMBDA_O, capacity=1024)
        win.grads.copy_(grad)
        win.m.copy_(m)
        win.v.copy_(v)
        win.step_dev.fill_(9)
        s.update(win=win)
    elif op == "densify":
        p, m, v, accum, denom, normals = _densify_inputs(case, seed)
        s.update(p=p, m=m, v=v, accum=accum, denom=denom, normals=normals,
                 ws=torch.empty(N.cgs_densify_workspace(case["n"]), dtype=torch.uint8, device="cuda"),
                 n_out=torch.zeros(1, dtype=torch.int64, device="cuda"),
                 out=[torch.zeros(N.cgs_param_count(2 * case["n"], case["sh_degree"]), device="cuda")
                      for _ in range(3)])                # room for every Gaussian to become two
    elif op == "points":
        p, m, v, xyz, rgb = _points_inputs(case, seed)
        total = N.cgs_param_count(case["n"] + case["points"], case["sh_degree"])
        s.update(p=p, m=m, v=v, xyz=xyz, rgb=rgb, out=[torch.empty(total, device="cuda") for _ in range(3)],
                 ws=torch.empty(N.cgs_points_workspace(case["points"]), dtype=torch.uint8, device="cuda"),
                 status=torch.zeros(1, dtype=torch.int32, device="cuda"))
    else:
        raise ValueError(op)
    return s


# --------------------------------------------------------------------- pass
def run(s):
    case = s["case"]
    op = case["op"]
    if op == "iter":
        win = s["win"]
        if case["graph"]:
            s["graph"].replay()
        else:
            win.forward()
            win.backward()
        return dict(loss=win.loss_view, img=win.img, depth=win.depth, t_final=win.t_final, grads=win.grads,
                    accum=win.accum, denom=win.denom, max_r2d=win.max_r2d)
    if op == "autograd":
        img, depth = RenderWindow.apply(s["params"], s["win"])
        loss = (img - s["rgb"]).abs().mean() + LAMBDA_DEPTH * ((depth - s["depth"]).abs() * s["valid"]).mean()
        return dict(loss=loss.detach(), img=img.detach(), depth=depth.detach(),
                    grads=torch.autograd.grad(loss, s["params"])[0])
    if op == "render":
        win = s["win"]
        win.forward(with_loss=False)
        return dict(img=win.img, depth=win.depth, t_final=win.t_final)
    if op == "ssim":
        N.cgs_ssim_loss(s["img"], s["rgb"], s["rendered"], s["depth"], s["count"], case["views"], s["cfg"],
                        s["weight"], case["lambda_ssim"], s["loss"], s["dimg"], s["ddepth"], s["ws"], s["status"])
        return dict(loss=s["loss"], dimg=s["dimg"], ddepth=s["ddepth"])
    if op == "adam":
        win = s["win"]
        win.optimizer_step()
        return dict(params=win.params, m=win.m, v=win.v, loss_o=win.loss_o)
    if op == "densify":
        n, deg = case["n"], case["sh_degree"]
        N.cgs_densify_plan(s["p"], n, deg, s["accum"], s["denom"], TAU_P, SCALE_THR, EPS_ALPHA, s["ws"], s["n_out"])
        n_out = int(s["n_out"].item())               # the new map's size, which its layout depends on
        N.cgs_densify_apply(s["p"], s["m"], s["v"], n, deg, s["ws"], s["normals"], n_out, *s["out"])
        return dict(n=n_out, params=s["out"][0], m=s["out"][1], v=s["out"][2])
    N.cgs_points_to_gaussians(s["p"], s["m"], s["v"], case["n"], case["sh_degree"], s["xyz"], s["rgb"],
                              case["points"], INIT_OPACITY, s["ws"], *s["out"], s["status"])
    return dict(params=s["out"][0], m=s["out"][1], v=s["out"][2])


def work(case):
    op = case["op"]
    if op == "ssim":
        px = case["width"] * case["height"] * case["views"]
        # images, targets and gradients of three channels; depth, target depth and gradient.
        # Two separable 11-tap blurs of five moments and three partials per value.
        return dict(bytes=px * (3 * 12 + 12), flops=px * 3 * (2 * 2 * 11 * 8 + 60))
    n, deg = case["n"], case["sh_degree"]
    P = (14 + 3 * ((deg + 1) ** 2 - 1)) * n
    if op == "adam":
        return dict(bytes=28 * P, flops=14 * P)
    if op == "densify":
        return dict(bytes=4 * (3 * P + 2 * n + 6 * n) + 4 * 3 * P, flops=40 * n)   # about as many come out
    if op == "points":
        k = case["points"]
        return dict(bytes=4 * (3 * P + 6 * k) + 4 * 3 * (P + P // n * k), flops=27 * 8 * k)
    # Windows: parameters in, images, depth and transmittance out; with a loss also targets in,
    # gradients and statistics out.  The blend evaluates about 400 (splat, pixel) pairs per
    # pixel for each Gaussian per pixel (150 on the largest window) at 13 operations, two
    # thirds of them blended at 11 more in the forward and 55 more in the backward.
    px = case["width"] * case["height"] * case["views"]
    pairs = 400.0 * min(0.4, n / (case["width"] * case["height"])) * px
    if op == "render":
        return dict(bytes=4 * P + 20 * px, flops=pairs * (13 + 0.66 * 11))
    return dict(bytes=8 * P + (20 + 16) * px + 24 * n, flops=pairs * (2 * 13 + 0.66 * 66))


# ------------------------------------------------------- values in 64 bits
def _sh_basis(d, deg):
    x, y, z = d.unbind(-1)
    xx, yy, zz = x * x, y * y, z * z
    pi = math.pi
    Y = [torch.full_like(x, 0.5 / math.sqrt(pi))]
    if deg >= 1:
        c = math.sqrt(3 / (4 * pi))
        Y += [-c * y, c * z, -c * x]
    if deg >= 2:
        c = 0.5 * math.sqrt(15 / pi)
        Y += [c * x * y, -c * y * z, 0.25 * math.sqrt(5 / pi) * (2 * zz - xx - yy), -c * x * z, 0.5 * c * (xx - yy)]
    if deg >= 3:
        a, b, c = 0.25 * math.sqrt(35 / (2 * pi)), 0.5 * math.sqrt(105 / pi), 0.25 * math.sqrt(21 / (2 * pi))
        Y += [-a * y * (3 * xx - yy), b * x * y * z, -c * y * (4 * zz - xx - yy),
              0.25 * math.sqrt(7 / pi) * z * (2 * zz - 3 * xx - 3 * yy), -c * x * (4 * zz - xx - yy),
              0.5 * b * z * (xx - yy), -a * x * (xx - 3 * yy)]
    return torch.stack(Y, -1)


def _split(P, n, deg):
    k = (deg + 1) ** 2
    sizes = [(n, 3), (n, 3), (n, 4), (n,), (n, 3), (n, k - 1, 3)]
    return [x.reshape(s) for x, s in zip(P.split([math.prod(s) for s in sizes]), sizes)]


def _rotation(q):
    w, x, y, z = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1).reshape(-1, 3, 3)


def _project(P, n, deg, cam, w, h):
    """One view's projected Gaussians: fields [n, 10] (u, v, A, B, C, opacity, z, r, g, b),
    radius [n] (0: culled) and tile rectangles."""
    means, ls, q, logit, dc, rest = _split(P, n, deg)
    R, t = cam[:9].reshape(3, 3), cam[9:12]
    fx, fy, cx, cy = cam[12:16]
    c = means @ R.T + t
    front = c[:, 2] > 0.2
    z = torch.where(front, c[:, 2], torch.ones_like(c[:, 2]))
    M = _rotation(q) * ls.exp()[:, None, :]
    S = M @ M.transpose(1, 2)
    lx, ly = 1.3 * 0.5 * w / fx, 1.3 * 0.5 * h / fy
    xc = torch.clamp(c[:, 0] / z, -lx, lx) * z
    yc = torch.clamp(c[:, 1] / z, -ly, ly) * z
    zero = torch.zeros_like(z)
    J = torch.stack([fx / z, zero, -fx * xc / z ** 2, zero, fy / z, -fy * yc / z ** 2], 1).reshape(-1, 2, 3)
    T = J @ R
    cov = T @ S @ T.transpose(1, 2)
    a, b, d = cov[:, 0, 0] + 0.3, cov[:, 0, 1], cov[:, 1, 1] + 0.3
    det = a * d - b * b
    u, v = fx * c[:, 0] / z + cx, fy * c[:, 1] / z + cy
    dirs = means + (R.T @ t)
    Y = _sh_basis(dirs / dirs.norm(dim=1, keepdim=True), deg)
    rgb = ((Y[:, :, None] * torch.cat([dc[:, None], rest], 1)).sum(1) + 0.5).clamp(min=0)
    rec = torch.cat([torch.stack([u, v, d / det, -b / det, a / det, torch.sigmoid(logit), c[:, 2]], 1), rgb], 1)
    with torch.no_grad():
        lam = 0.5 * (a + d) + (0.25 * (a - d) ** 2 + b * b).clamp(min=0.1).sqrt()
        r = (3 * lam.sqrt()).ceil()
        tx, ty = (w + 15) // 16, (h + 15) // 16
        fu, fv = u.floor(), v.floor()
        rect = [((fu - r) / 16).floor().clamp(0, tx), ((fu + r + 15) / 16).floor().clamp(0, tx),
                ((fv - r) / 16).floor().clamp(0, ty), ((fv + r + 15) / 16).floor().clamp(0, ty)]
        seen = front & (det > 0) & (rect[1] > rect[0]) & (rect[3] > rect[2])
    return rec, torch.where(seen, r, torch.zeros_like(r)), rect


def _blend(rec, xs, ys):
    """Front-to-back blend of depth-sorted fields [L, 10] at pixels [p]: colour, depth, T."""
    dx, dy = rec[:, 0:1] - xs, rec[:, 1:2] - ys
    power = -0.5 * (rec[:, 2:3] * dx * dx + rec[:, 4:5] * dy * dy) - rec[:, 3:4] * dx * dy
    alpha = (rec[:, 5:6] * power.exp()).clamp(max=0.99)
    alpha = torch.where((power <= 0) & (alpha >= 1 / 255), alpha, torch.zeros_like(alpha))
    with torch.no_grad():
        live = (1 - alpha).cumprod(0) >= 1e-4
    alpha = torch.where(live, alpha, torch.zeros_like(alpha))
    T = (1 - alpha).cumprod(0)
    wgt = alpha * torch.cat([torch.ones_like(T[:1]), T[:-1]])
    return rec[:, 7:10].T @ wgt, rec[:, 6] @ wgt, T[-1]


def _exact_views(case, P, cams, loss_of):
    """(img, depth, T, parameter gradient or None, per-view centre gradients, radii): the
    pixel gradients come from loss_of(img, depth), evaluated on the rendered views."""
    n, deg, w, h, V = (case[k] for k in ("n", "sh_degree", "width", "height", "views"))
    bg = torch.tensor(BG, dtype=torch.float32, device="cuda").double()
    img = bg[None, :, None, None].expand(V, 3, h, w).clone()
    depth = torch.zeros(V, h, w, dtype=torch.float64, device="cuda")
    tfin = torch.ones(V, h, w, dtype=torch.float64, device="cuda")
    P = P.double().requires_grad_(loss_of is not None)

    def tiles(rec, radius, rect):
        near = torch.argsort(rec[:, 6].detach(), stable=True)
        near = near[radius[near] > 0]
        x0, x1, y0, y1 = (r[near] for r in rect)
        for ty in range((h + 15) // 16):
            row = (y0 <= ty) & (y1 > ty)
            near_row, rx0, rx1 = near[row], x0[row], x1[row]
            ys, ye = 16 * ty, min(h, 16 * ty + 16)
            for tx in range((w + 15) // 16):
                ids = near_row[(rx0 <= tx) & (rx1 > tx)]
                if ids.numel() == 0:
                    continue
                xs, xe = 16 * tx, min(w, 16 * tx + 16)
                yy, xx = torch.meshgrid(torch.arange(ys, ye, device="cuda", dtype=torch.float64),
                                        torch.arange(xs, xe, device="cuda", dtype=torch.float64), indexing="ij")
                yield ids, (slice(ys, ye), slice(xs, xe)), xx.reshape(-1), yy.reshape(-1)

    views = [_project(P, n, deg, cams[v].double(), w, h) for v in range(V)]
    with torch.no_grad():
        for v, (rec, radius, rect) in enumerate(views):
            for ids, (sy, sx), xx, yy in tiles(rec, radius, rect):
                c, d, T = _blend(rec[ids], xx, yy)
                shape = img[v, 0, sy, sx].shape
                img[v, :, sy, sx] = (c + T * bg[:, None]).reshape(3, *shape)
                depth[v, sy, sx], tfin[v, sy, sx] = d.reshape(shape), T.reshape(shape)
    if loss_of is None:
        return img, depth, tfin, None, None, None
    leaf_i, leaf_d = img.clone().requires_grad_(True), depth.clone().requires_grad_(True)
    gi, gd = torch.autograd.grad(loss_of(leaf_i, leaf_d).sum(), [leaf_i, leaf_d])
    grecs = []
    for v, (rec, radius, rect) in enumerate(views):
        grec = torch.zeros_like(rec)
        for ids, (sy, sx), xx, yy in tiles(rec.detach(), radius, rect):
            sub = rec.detach()[ids].requires_grad_(True)
            c, d, T = _blend(sub, xx, yy)
            s = ((c + T * bg[:, None]) * gi[v, :, sy, sx].reshape(3, -1)).sum() + (d * gd[v, sy, sx].reshape(-1)).sum()
            grec.index_add_(0, ids, torch.autograd.grad(s, sub)[0])
        grecs.append(grec)
    total = torch.autograd.grad([v[0] for v in views], P, grecs)[0]
    return img, depth, tfin, total, [x[:, :2] for x in grecs], [v[1] for v in views]


def _blur(x):
    k = torch.arange(-5, 6, device="cuda", dtype=torch.float64)
    k = torch.exp(-k * k / 4.5)
    k = k / k.sum()
    x = torch.nn.functional.conv2d(x, k.reshape(1, 1, 1, 11), padding=(0, 5))
    return torch.nn.functional.conv2d(x, k.reshape(1, 1, 11, 1), padding=(5, 0))


def _loss(img, depth, rgb, tdepth, weight, lam):
    """Per-view loss of Eq. 9 plus the depth term."""
    rgb, tdepth = rgb.double(), tdepth.double()
    V, _, h, w = img.shape
    L = (1 - lam) * (img - rgb).abs().mean((1, 2, 3))
    if lam > 0:
        x, y = img.reshape(-1, 1, h, w), rgb.reshape(-1, 1, h, w)
        mx, my = _blur(x), _blur(y)
        sx, sy, sxy = _blur(x * x) - mx * mx, _blur(y * y) - my * my, _blur(x * y) - mx * my
        S = (2 * mx * my + 1e-4) * (2 * sxy + 9e-4) / ((mx * mx + my * my + 1e-4) * (sx + sy + 9e-4))
        L = L + lam * (1 - S.reshape(V, -1).mean(1))
    valid = tdepth > 0
    L = L + LAMBDA_DEPTH * ((depth - tdepth).abs() * valid).sum((1, 2)) / valid.sum((1, 2))
    return weight.double() * L


def exact(case, seed):
    op = case["op"]
    if op in ("iter", "autograd", "render"):
        tiles = case["views"] * ((case["width"] + 15) // 16) * ((case["height"] + 15) // 16)
        if tiles * (1 if op == "render" else 4) > 14500:
            return None                                   # the tile-by-tile evaluation takes too long
        p, cams, rgb, tdepth, weight = _window_inputs(case, seed)
        if op == "render":
            img, depth, tfin = _exact_views(case, p, cams, None)[:3]
            return dict(img=img, depth=depth, t_final=tfin)
        if op == "autograd":
            valid = tdepth > 0

            def own(i, d):
                return (i - rgb.double()).abs().mean() + LAMBDA_DEPTH * ((d - tdepth.double()).abs() * valid).mean()
            img, depth, _, grads, _, _ = _exact_views(case, p, cams, own)
            return dict(loss=own(img, depth), img=img, depth=depth, grads=grads)

        def eq9(i, d):
            return _loss(i, d, rgb, tdepth, weight, case["lambda_ssim"])
        img, depth, tfin, grads, gc, radii = _exact_views(case, p, cams, eq9)
        half = torch.tensor([0.5 * case["width"], 0.5 * case["height"]], dtype=torch.float64, device="cuda")
        return dict(loss=eq9(img, depth), img=img, depth=depth, t_final=tfin, grads=grads,
                    accum=sum((g * half).norm(dim=1) for g in gc), denom=sum((r > 0).double() for r in radii),
                    max_r2d=torch.stack(radii).amax(0))
    if op == "ssim":
        s = prepare(case, seed)
        img, d = s["img"].double().requires_grad_(True), s["rendered"].double().requires_grad_(True)
        loss = _loss(img, d, s["rgb"], s["depth"], s["weight"], case["lambda_ssim"])
        gi, gd = torch.autograd.grad(loss.sum(), [img, d])
        return dict(loss=loss.detach(), dimg=gi, ddepth=gd)
    n, deg = case["n"], case["sh_degree"]
    if op == "adam":
        p, g, m, v = (x.double() for x in _adam_inputs(case, seed))
        lr = torch.cat([torch.full_like(x.reshape(-1), l) for x, l in zip(_split(p, n, deg), LR)])
        o = torch.sigmoid(p[10 * n: 11 * n])
        g[10 * n: 11 * n] += LAMBDA_O / n * o * (1 - o)
        m = BETAS[0] * m + (1 - BETAS[0]) * g
        v = BETAS[1] * v + (1 - BETAS[1]) * g * g
        p = p - lr * (m / (1 - BETAS[0] ** 10)) / ((v / (1 - BETAS[1] ** 10)).sqrt() + EPS)
        return dict(params=p, m=m, v=v, loss_o=(LAMBDA_O * o.mean()).reshape(1))
    if op == "densify":
        p, m, v, accum, denom, normals = _densify_inputs(case, seed)
        parts, mom, var = (_split(x, n, deg) for x in (p, m, v))
        grad = torch.where(denom > 0, accum / denom, torch.zeros_like(accum))
        high = grad >= torch.tensor(TAU_P, dtype=torch.float32, device="cuda")
        small = parts[1].amax(1) <= torch.tensor(math.log(SCALE_THR), dtype=torch.float32, device="cuda")
        prune = parts[3] < torch.tensor(math.log(EPS_ALPHA / (1 - EPS_ALPHA)), dtype=torch.float32, device="cuda")
        copies = torch.where(prune, 0, torch.where(high, 2, 1))
        src = torch.repeat_interleave(torch.arange(n, device="cuda"), copies)
        child = torch.cat([torch.zeros_like(src[:1]), (src[1:] == src[:-1]).long()])
        split = (high & ~small)[src]
        fresh = (split | (child == 1))
        out = [x.double()[src] for x in parts]
        off = _rotation(parts[2].double()) @ (parts[1].double().exp()[:, :, None] * normals.double().transpose(1, 2))
        off = off[src, :, child]
        out[0] = torch.where(split[:, None], out[0] + off, out[0])
        out[1] = torch.where(split[:, None], out[1] - math.log(1.6), out[1])
        keep = [[torch.where(fresh.reshape(-1, *[1] * (x.dim() - 1)), 0.0, x.double()[src]) for x in part]
                for part in (mom, var)]
        flat = [torch.cat([x.reshape(-1) for x in part]) for part in (out, *keep)]
        room = 2 * p.numel()
        flat = [torch.nn.functional.pad(x, (0, room - x.numel())) for x in flat]
        return dict(n=None, params=flat[0], m=flat[1], v=flat[2])
    p, m, v, xyz, rgb = _points_inputs(case, seed)
    x, k = xyz.double(), case["points"]
    near = []
    for i in range(0, k, 2048):                           # exact three nearest others, brute force
        d2 = sum((x[i:i + 2048, a:a + 1] - x[None, :, a]) ** 2 for a in range(3))
        rows = torch.arange(d2.shape[0], device="cuda")
        d2[rows, i + rows] = math.inf
        near.append(d2.topk(3, dim=1, largest=False)[0].mean(1))
    ls = 0.5 * torch.cat(near).clamp(min=1e-7).log()
    unit = torch.tensor([1.0, 0, 0, 0], dtype=torch.float64, device="cuda")
    new = [x, ls[:, None].expand(k, 3), unit.expand(k, 4), torch.full_like(ls, math.log(INIT_OPACITY / (1 - INIT_OPACITY))),
           (rgb.double() - 0.5) / Y00, torch.zeros(k, (deg + 1) ** 2 - 1, 3, dtype=torch.float64, device="cuda")]

    def joined(flat, tail):
        return torch.cat([torch.cat([a.double(), b]).reshape(-1) for a, b in zip(_split(flat, n, deg), tail)])
    none = [torch.zeros_like(b) for b in new]
    return dict(params=joined(p, new), m=joined(m, none), v=joined(v, none))
