"""Timed cases of the Beta rasterizer: what a program using this package has it do.

A training program renders one view or a batch of views of a scene, takes the
gradient of an image loss and updates the parameters; a viewer renders single
frames.  Every case goes through the package's public entry points
(`Rasterizer`, `render`, `BatchedStep`, `BetaAdam`) the way such a program
calls them, on seeded synthetic scenes of the recipes in `scenes.py` (drawn on
the GPU here, so that a scene of millions of primitives takes no time).

listed()             the named cases
draw(rng)            one more case of the same ranges
prepare(case, seed)  the inputs and handles a program holds before the call
run(state)           one pass through the public entry points
work(case)           bytes and flops of one pass that no implementation avoids
exact(case, seed)    the outputs in 64 bits by plain torch (None: too large)
"""
import math

import torch

from paper_2501_18630_gb300 import _lib, batched, optim, render, scenes

DEV = "cuda"
# a batch of views in the four resolutions of the mixed-resolution workload
MIXED = "mixed"


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def _case(name, kind, **kw):
    c = {"name": name, "kind": kind}
    c.update(kw)
    return c


def listed():
    return [
        # one small preview frame, forward only: launches and latency count
        _case("render_4k_256x256", "render", scene="cube", n=4096, lobes=1, views=1, width=256, height=256,
              tile_w=16, tile_h=16, batch_s=256, blur=0.0, color_mode=0),
        # a viewer's frame of a trained scene of about three million primitives
        _case("render_3100k_1080p", "render", scene="sheets", n=3_100_000, lobes=2, views=1, width=1920, height=1080,
              tile_w=16, tile_h=16, batch_s=256, blur=0.0, color_mode=0),
        # one training view through torch.autograd, early in training (odd width)
        _case("autograd_200k_1297x840", "autograd", scene="gmm", n=200_000, lobes=2, views=1, width=1297, height=840,
              tile_w=16, tile_h=16, batch_s=256, blur=0.0, color_mode=0),
        # one training view through torch.autograd at full size
        _case("autograd_1m_1080p", "autograd", scene="sheets", n=1_000_000, lobes=3, views=1, width=1920, height=1080,
              tile_w=16, tile_h=16, batch_s=256, blur=0.0, color_mode=0),
        # the training iteration of the paper's loss: forward, L1 + DSSIM, backward
        _case("train_dssim_500k_1297x840", "train", scene="sheets", n=500_000, lobes=2, views=1, width=1297,
              height=840, tile_w=16, tile_h=16, batch_s=256, blur=0.0, color_mode=0),
        # a small batch of odd-sized views, the captured step with its defaults (persistent, 16x16 tiles)
        _case("batch_100k_4x641x479", "batch", scene="gmm", n=99_991, lobes=1, views=4, width=641, height=479,
              tile_w=16, tile_h=16, batch_s=256, blur=0.0, color_mode=0, persistent=True, fused=True),
        # the benchmark's captured step: 16 views of 1080p
        _case("batch_1m_16x1080p", "batch", scene="sheets", n=1_000_000, lobes=3, views=16, width=1920, height=1080,
              tile_w=16, tile_h=8, batch_s=64, blur=0.0, color_mode=0, persistent=False, fused=True),
        # the captured step over 16 views of four resolutions
        _case("batch_3m_16xmixed", "batch", scene="sheets", n=3_000_000, lobes=3, views=16, width=0, height=0,
              tile_w=8, tile_h=8, batch_s=64, blur=0.0, color_mode=0, persistent=False, fused=True),
        # the largest captured step: 8 views of 4K, two raster launches with hit masks
        _case("batch_6m_8x4k", "batch", scene="sheets", n=6_000_000, lobes=3, views=8, width=3840, height=2160,
              tile_w=16, tile_h=8, batch_s=64, blur=0.0, color_mode=0, persistent=False, fused=False),
        # the image loss on its own, on a batch of rendered views
        _case("dssim_16x1080p", "dssim", views=16, width=1920, height=1080, ssim=0.2),
        # the optimiser step of the full-size scene
        _case("adam_1m", "adam", n=1_000_000, lobes=3),
        # respawning the dead primitives of the full-size scene
        _case("relocate_1m", "relocate", n=1_000_000, lobes=3, dead=0.03),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# (tile_w, tile_h, batch_s) that users pick: the default, the autotuner's candidates, the other shapes
_TILES = [(16, 16, 256), (16, 16, 256), (16, 16, 128), (16, 8, 64), (16, 8, 64), (16, 8, 128), (8, 8, 64), (8, 8, 128),
          (32, 16, 128), (8, 4, 64)]


def draw(rng):
    kind = rng.choice(["render", "render", "autograd", "autograd", "train", "batch", "batch", "batch", "dssim", "adam",
                       "relocate"])
    c = {"kind": kind}
    if kind == "adam":
        c.update(n=_log_int(rng, 4000, 4_000_000), lobes=rng.randint(0, 4))
        return c
    if kind == "relocate":
        c.update(n=_log_int(rng, 4000, 4_000_000), lobes=rng.randint(0, 4), dead=round(rng.uniform(0.0005, 0.08), 4))
        return c
    if kind == "dssim":
        w = _log_int(rng, 200, 2600)
        c.update(views=rng.randint(1, 8), width=w, height=max(1, int(w * rng.uniform(0.5, 0.8))),
                 ssim=round(rng.uniform(0.05, 0.5), 3))
        return c
    scene = rng.choice(["cube", "gmm", "sheets", "sheets"])
    n = _log_int(rng, 2000, {"cube": 20_000, "gmm": 500_000, "sheets": 3_000_000}[scene])
    w = _log_int(rng, 160, 2600)
    tw, th, s = rng.choice(_TILES)
    c.update(scene=scene, n=n, lobes=rng.randint(0, 4), views=1, width=w, height=max(1, int(w * rng.uniform(0.5, 0.8))),
             tile_w=tw, tile_h=th, batch_s=s, blur=rng.choice([0.0, 0.0, 0.0, 0.3]), color_mode=rng.choice([0, 0, 0, 1, 2]))
    if c["lobes"] == 0 and c["color_mode"] == 2:
        c["color_mode"] = 0                   # the lobes alone: there are some
    if kind == "batch":
        c["views"] = rng.randint(2, 12)
        c["persistent"] = rng.random() < 0.5
        c["fused"] = rng.random() < 0.7
        c["n"] = min(n, 1_500_000)
        if rng.random() < 0.3:
            c["width"] = c["height"] = 0      # views of the four mixed resolutions
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

class _Draws:
    """Seeded float32 draws on the GPU."""

    def __init__(self, seed, stream=0):
        self.g = torch.Generator(device=DEV)
        self.g.manual_seed(int(seed) * 8191 + stream)

    def normal(self, *shape):
        return torch.randn(*shape, generator=self.g, device=DEV)

    def uniform(self, *shape, lo=0.0, hi=1.0):
        return torch.rand(*shape, generator=self.g, device=DEV) * (hi - lo) + lo

    def index(self, k, n):
        return torch.randint(0, k, (n,), generator=self.g, device=DEV)


def _frames_to_quats(R):
    """Rotation matrices (n, 3, 3) -> unit quaternions (n, 4), w x y z."""
    d = torch.diagonal(R, dim1=1, dim2=2)
    w = 0.5 * torch.sqrt(torch.clamp(1.0 + d[:, 0] + d[:, 1] + d[:, 2], min=0.0))
    x = 0.5 * torch.sqrt(torch.clamp(1.0 + d[:, 0] - d[:, 1] - d[:, 2], min=0.0))
    y = 0.5 * torch.sqrt(torch.clamp(1.0 - d[:, 0] + d[:, 1] - d[:, 2], min=0.0))
    z = 0.5 * torch.sqrt(torch.clamp(1.0 - d[:, 0] - d[:, 1] + d[:, 2], min=0.0))
    x = torch.copysign(x, R[:, 2, 1] - R[:, 1, 2])
    y = torch.copysign(y, R[:, 0, 2] - R[:, 2, 0])
    z = torch.copysign(z, R[:, 1, 0] - R[:, 0, 1])
    q = torch.stack([w, x, y, z], 1)
    return q / q.norm(dim=1, keepdim=True)


def _unit(v):
    return v / v.norm(dim=1, keepdim=True)


def _scene_planes(scene, n, lobes, seed):
    """Parameter planes (15 + 6 M, pitch) of a scene recipe of scenes.py."""
    d = _Draws(seed, 1)
    pl = torch.zeros(scenes.n_planes(lobes), scenes.round_pitch(n), device=DEV)
    pl[scenes.P_QUAT] = 1.0
    quat = _unit(d.normal(n, 4))
    if scene == "cube":
        mean, ls = d.uniform(3, n, lo=-1.0, hi=1.0), -3.5 + 0.4 * d.normal(3, n)
        op_sd, b_sd = 1.0, 0.5
    elif scene == "gmm":
        centre, sig = d.uniform(64, 3, lo=-2.0, hi=2.0), d.uniform(64, lo=0.05, hi=0.3)
        comp = d.index(64, n)
        mean = (centre[comp] + sig[comp, None] * d.normal(n, 3)).clamp(-2.0, 2.0).T
        ls = -4.5 + 0.5 * d.normal(3, n)
        op_sd, b_sd = 1.5, 0.7
    else:
        k = 256
        centre, normal, radius = d.uniform(k, 3, lo=-1.5, hi=1.5), _unit(d.normal(k, 3)), d.uniform(k, lo=0.3, hi=0.8)
        helper = torch.where(normal[:, :1].abs() < 0.9, torch.tensor([[1.0, 0.0, 0.0]], device=DEV),
                             torch.tensor([[0.0, 1.0, 0.0]], device=DEV))
        e1 = _unit(torch.linalg.cross(normal, helper))
        e2 = torch.linalg.cross(normal, e1)
        s = d.index(k, n)
        rho, ang = d.uniform(n).sqrt() * radius[s], d.uniform(n, hi=2.0 * math.pi)
        mean = (centre[s] + (rho * ang.cos())[:, None] * e1[s] + (rho * ang.sin())[:, None] * e2[s]
                + 0.005 * d.normal(n)[:, None] * normal[s]).T
        ls = -5.0 + 0.6 * d.normal(3, n)
        ls[2] -= math.log(10.0)
        tw = d.uniform(n, hi=2.0 * math.pi)
        u = tw.cos()[:, None] * e1[s] + tw.sin()[:, None] * e2[s]
        v = -tw.sin()[:, None] * e1[s] + tw.cos()[:, None] * e2[s]
        quat = _frames_to_quats(torch.stack([u, v, normal[s]], 2))
        op_sd, b_sd = 1.5, 0.7
    pl[0:3, :n] = mean
    pl[3:6, :n] = ls
    pl[6:10, :n] = quat.T
    pl[10, :n] = op_sd * d.normal(n)
    pl[11, :n] = b_sd * d.normal(n)
    pl[12:15, :n] = d.uniform(3, n)
    for m in range(lobes):
        b = scenes.P_LOBES + scenes.LOBE_STRIDE * m
        pl[b, :n] = torch.arccos(d.uniform(n, lo=-1.0, hi=1.0))
        pl[b + 1, :n] = d.uniform(n, hi=2.0 * math.pi)
        pl[b + 2, :n] = 0.5 * d.normal(n)
        pl[b + 3:b + 6, :n] = d.uniform(3, n, hi=0.5)
    return pl


def _sizes(case):
    if case["width"]:
        return [(case["width"], case["height"])] * case["views"]
    return [scenes.MIXED_SIZES[k // 4 % 4] for k in range(case["views"])]


def _cameras(case):
    if case["scene"] == "cube" and case["views"] == 1:
        R, t = scenes.look_at((0.0, 0.0, -3.0))
        return [scenes.pinhole(R, t, w, h) for w, h in _sizes(case)]
    v = case["views"]
    return [scenes.ring_camera(4.0, 15.0, 2.0 * math.pi * k / v, w, h) for k, (w, h) in enumerate(_sizes(case))]


def _opts(case):
    return _lib.default_opts(tile_w=case["tile_w"], tile_h=case["tile_h"], batch_s=case["batch_s"],
                             blur_eps=case["blur"], color_mode=case["color_mode"])


def _pixels(case):
    return sum(w * h for w, h in _sizes(case))


def _target(case, seed):
    """Target images, U[0, 1] per value as scenes.target_images draws them (planar, view after view)."""
    return _Draws(seed, 2).uniform(3 * _pixels(case))


def _image_pair(case, seed):
    """A batch of smooth target images and rendered ones near them."""
    d = _Draws(seed, 3)
    v, h, w = case["views"], case["height"], case["width"]
    low = d.uniform(v, 3, max(2, h // 24), max(2, w // 24))
    y = torch.nn.functional.interpolate(low, size=(h, w), mode="bilinear", align_corners=False)
    y = (y + 0.03 * d.normal(v, 3, h, w)).clamp(0.0, 1.0)
    x = (y + 0.08 * d.normal(v, 3, h, w)).clamp(0.0, 1.0)
    return x.reshape(-1).contiguous(), y.reshape(-1).contiguous()


def _optim_inputs(case, seed):
    """Parameters, gradients, moments and noise in the middle of a training run:
    about a third of the primitives had no gradient in the last step."""
    n, m = case["n"], case["lobes"]
    d = _Draws(seed, 4)
    planes = _scene_planes("sheets", n, m, seed)
    shape = planes.shape
    seen = (d.uniform(1, shape[1]) < 0.65).float()
    grad = 1e-5 * d.normal(*shape) * seen
    mom = 5e-6 * d.normal(*shape)
    var = (1e-5 * d.normal(*shape)) ** 2
    eta = d.normal(3, shape[1])
    return planes, grad, mom, var, eta


def _adam_state(case, seed):
    planes, grad, mom, var, eta = _optim_inputs(case, seed)
    opt = optim.BetaAdam(planes, case["n"], case["lobes"])
    opt.m.copy_(mom)
    opt.v.copy_(var)
    opt.t = 500
    return planes, grad, eta, opt


def prepare(case, seed):
    kind = case["kind"]
    st = {"kind": kind}
    if kind == "adam":
        st["planes"], st["grad"], st["eta"], st["opt"] = _adam_state(case, seed)
        return st
    if kind == "relocate":
        planes, _, _, opt = _adam_state(case, seed)
        d = _Draws(seed, 5)
        n = case["n"]
        dead = d.uniform(n) < case["dead"]
        planes[scenes.P_OPACITY, :n] = torch.where(dead, -7.0 + d.normal(n).clamp(-3, 1), planes[scenes.P_OPACITY, :n])
        st.update(planes=planes, opt=opt, logit=planes[scenes.P_OPACITY].clone(),
                  rnd=torch.randint(-2 ** 31, 2 ** 31, (n,), dtype=torch.int32, device=DEV, generator=d.g))
        return st
    if kind == "dssim":
        x, y = _image_pair(case, seed)
        R, t = scenes.look_at((0.0, 0.0, -3.0))
        cams = [scenes.pinhole(R, t, case["width"], case["height"]) for _ in range(case["views"])]
        rast = render.Rasterizer(32, 32, 0, cams)
        rast.color.copy_(x)
        st.update(rast=rast, target=y, ssim=case["ssim"])
        return st
    n, m = case["n"], case["lobes"]
    planes = _scene_planes(case["scene"], n, m, seed)
    cams = _cameras(case)
    if kind == "batch":
        step = batched.BatchedStep(planes, n, m, cams, _target(case, seed), opts=_opts(case),
                                   persistent=case["persistent"], fused=case["fused"])
        step.capture()
        st["step"] = step
        return st
    rast = render.Rasterizer(n, planes.shape[1], m, cams, opts=_opts(case))
    rast.forward(planes)          # the first frame sizes the pair buffers
    st.update(rast=rast, planes=planes)
    if kind == "autograd":
        planes.requires_grad_(True)
        st["target"] = _target(case, seed)
    elif kind == "train":
        st["target"] = _target(case, seed)
        st["grad"] = torch.zeros_like(planes)
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(st):
    kind = st["kind"]
    if kind == "render":
        rast = st["rast"]
        return {"color": rast.forward(st["planes"]), "T": rast.T_final}
    if kind == "autograd":
        planes = st["planes"]
        planes.grad = None
        color = render.render(planes, st["rast"])
        loss = (color - st["target"]).abs().mean()
        loss.backward()
        return {"color": color, "loss": loss, "grad": planes.grad}
    if kind == "train":
        rast, planes = st["rast"], st["planes"]
        color = rast.forward(planes, check_capacity=False)
        loss, dl = rast.dssim_loss(st["target"], 0.2)
        grad = rast.backward(planes, dl, st["grad"])
        return {"color": color, "loss": loss, "dcolor": dl, "grad": grad}
    if kind == "batch":
        step = st["step"]
        step.step()
        return {"color": step.rast.color, "loss": step.loss, "grad": step.grad}
    if kind == "dssim":
        loss, dl = st["rast"].dssim_loss(st["target"], st["ssim"])
        return {"loss": loss, "dcolor": dl}
    opt = st["opt"]
    if kind == "adam":
        opt.step(st["planes"], st["grad"], eta=st["eta"])
        return {"planes": st["planes"], "m": opt.m, "v": opt.v, "reg": opt.reg_loss}
    # relocation: the optimiser steps between two calls have left primitives
    # dead again (a copy of the opacity plane stands in for those steps)
    st["planes"][scenes.P_OPACITY].copy_(st["logit"])
    count, src = opt.relocate(st["planes"], rnd=st["rnd"])
    return {"planes": st["planes"], "m": opt.m, "v": opt.v, "count": count, "src": src}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def work(case):
    """Inputs read once, outputs written once; flops of the arithmetic per
    primitive and view, per pixel and per filter tap (compositing depends on
    the scene and is left out of the flops)."""
    kind = case["kind"]
    if kind == "dssim":
        v = 3 * case["views"] * case["width"] * case["height"]
        return {"bytes": 12 * v, "flops": v * (2 * 2 * 11 * 7 + 40)}
    p = 4 * scenes.n_planes(case["lobes"])
    n = case["n"]
    if kind == "adam":
        return {"bytes": n * (7 * p + 12), "flops": n * (p // 4) * 14}
    if kind == "relocate":
        # opacity logits and random words read, sources written, the dead
        # primitives' parameters and moments copied or zeroed
        return {"bytes": n * 12 + case["dead"] * n * 4 * p, "flops": n * 20}
    px, v = _pixels(case), case["views"]
    b, f = n * p + px * 12, n * v * 300
    if kind == "render":
        return {"bytes": b + px * 4, "flops": f}
    b += px * 12 + n * p          # target read, gradients written
    if kind == "train":
        return {"bytes": b + px * 12, "flops": 2 * f + 3 * px * (2 * 2 * 11 * 7 + 40)}
    return {"bytes": b, "flops": 2 * f}


# ---------------------------------------------------------------------------
# 64-bit values by plain torch
# ---------------------------------------------------------------------------

_T_EPS, _ALPHA_MAX = 2.0 ** -19, 0.99
_BLOCK = 32              # pixels of a block's side; every block composites the primitives whose box meets it


def _project64(p, lobes, cam, blur, mode):
    """Per primitive: mean2d (2), whitening rows (p, q1, q2), log opacity, beta,
    colour (3) as columns, and the half extents and keep mask (no gradient)."""
    R = torch.as_tensor(cam.R, dtype=torch.float64, device=DEV)
    t = torch.as_tensor(cam.t, dtype=torch.float64, device=DEV)
    tc = R @ p[0:3] + t[:, None]
    keep = tc[2].detach() > cam.near
    z = torch.where(keep, tc[2], torch.ones_like(tc[2]))
    fx, fy = cam.fx, cam.fy
    s = torch.exp(p[3:6])
    q = p[6:10] / p[6:10].norm(dim=0, keepdim=True)
    w, x, y, zq = q
    Rq = torch.stack([torch.stack([1 - 2 * (y * y + zq * zq), 2 * (x * y - w * zq), 2 * (x * zq + w * y)]),
                      torch.stack([2 * (x * y + w * zq), 1 - 2 * (x * x + zq * zq), 2 * (y * zq - w * x)]),
                      torch.stack([2 * (x * zq - w * y), 2 * (y * zq + w * x), 1 - 2 * (x * x + y * y)])])
    A = torch.einsum("ij,jkn->ikn", R, Rq)
    M0 = (fx / z * A[0] - fx * tc[0] / z ** 2 * A[2]) * s
    M1 = (fy / z * A[1] - fy * tc[1] / z ** 2 * A[2]) * s
    a, b, c = (M0 * M0).sum(0) + blur, (M0 * M1).sum(0), (M1 * M1).sum(0) + blur
    m01, m02, m12 = M0[0] * M1[1] - M0[1] * M1[0], M0[0] * M1[2] - M0[2] * M1[0], M0[1] * M1[2] - M0[2] * M1[1]
    det = m01 ** 2 + m02 ** 2 + m12 ** 2 + blur * (a + c - blur)
    keep = keep & (det.detach() > 0) & (a.detach() > 0)
    a1, d1 = torch.where(keep, a, torch.ones_like(a)), torch.where(keep, det, torch.ones_like(det))
    pp = a1.rsqrt()
    isd = d1.rsqrt()
    q1, q2 = a1 * pp * isd, -b * pp * isd
    col = p[12:15] if mode != 2 else torch.zeros_like(p[12:15])
    if lobes and mode != 1:
        pos = -(R.T @ t)
        dirv = p[0:3] - pos[:, None]
        dirv = dirv / dirv.norm(dim=0, keepdim=True)
        for m in range(lobes):
            L = p[15 + 6 * m:21 + 6 * m]
            rm = torch.stack([L[0].sin() * L[1].cos(), L[0].sin() * L[1].sin(), L[0].cos()])
            dot = (rm * dirv).sum(0)
            on = dot.detach() > 0
            wgt = torch.where(on, torch.where(on, dot, torch.ones_like(dot)) ** (4 * torch.exp(L[2])), torch.zeros_like(dot))
            col = col + wgt * L[3:6]
    rec = torch.cat([(fx * tc[0] / z + cam.cx)[None], (fy * tc[1] / z + cam.cy)[None], pp[None], q1[None], q2[None],
                     torch.nn.functional.logsigmoid(p[10])[None], 4 * torch.exp(p[11])[None], col])
    # depth key: camera z in fp32, products and sums rounded in this order
    m32, Rf, tf = p[0:3].detach().float(), [float(v) for v in R[2]], float(t[2])
    key = m32[0] * Rf[0] + m32[1] * Rf[1]
    key = key + m32[2] * Rf[2]
    key = key + tf
    return rec, a.detach().clamp_min(0).sqrt(), c.detach().clamp_min(0).sqrt(), key, keep


def _blocks(rec, ex, ey, key, keep, w, h):
    """(x0, y0, x1, y1, primitives in depth order) of every pixel block that a primitive meets."""
    mx, my = rec[0].detach(), rec[1].detach()
    order = torch.nonzero(keep).squeeze(1)
    order = order[torch.sort(key[order], stable=True)[1]]
    lo_x, hi_x = (mx - ex - 1)[order], (mx + ex + 1)[order]
    lo_y, hi_y = (my - ey - 1)[order], (my + ey + 1)[order]
    for y0 in range(0, h, _BLOCK):
        y1 = min(h, y0 + _BLOCK)
        row = (lo_y <= y1) & (hi_y >= y0)
        ro, rl, rh = order[row], lo_x[row], hi_x[row]
        for x0 in range(0, w, _BLOCK):
            x1 = min(w, x0 + _BLOCK)
            ids = ro[(rl <= x1) & (rh >= x0)]
            yield x0, y0, x1, y1, ids


def _composite64(r, x0, y0, x1, y1):
    """(3, pixels) colour and (pixels) transmittance of one block from its records (10, k) in depth order."""
    ys, xs = torch.meshgrid(torch.arange(y0, y1, device=DEV, dtype=torch.float64) + 0.5,
                            torch.arange(x0, x1, device=DEV, dtype=torch.float64) + 0.5, indexing="ij")
    dx, dy = xs.reshape(-1, 1) - r[0], ys.reshape(-1, 1) - r[1]
    u, v = r[2] * dx, r[4] * dx + r[3] * dy
    x = 1.0 - (u * u + v * v)
    on = x.detach() > 0
    al = torch.where(on, torch.exp(r[6] * torch.log(torch.where(on, x, torch.ones_like(x))) + r[5]), torch.zeros_like(x))
    al = al.clamp(max=_ALPHA_MAX)
    T = torch.cumprod(1.0 - al, 1)
    before = torch.cat([torch.ones_like(T[:, :1]), T[:, :-1]], 1)
    live = before.detach() >= _T_EPS
    wgt = torch.where(live, al * before, torch.zeros_like(al))
    stop = live.sum(1) - 1
    return (wgt @ r[7:10].T).T, T.gather(1, stop[:, None])[:, 0]


def _render64(planes, case, cams, want_grad, dcolor=None, target=None):
    """Colour and transmittance of every view; with want_grad the gradient of
    the raw parameters for dL/dcolor (given, or the L1 loss's)."""
    p = planes[:, :case["n"]].double()
    colors, Ts, grad = [], [], torch.zeros_like(p)
    off = 0
    for cam in cams:
        w, h = cam.width, cam.height
        with torch.enable_grad():
            leaf = p.clone().requires_grad_(want_grad)
            rec, ex, ey, key, keep = _project64(leaf, case["lobes"], cam, case["blur"], case["color_mode"])
        C, T = torch.zeros(3, h, w, dtype=torch.float64, device=DEV), torch.ones(h, w, dtype=torch.float64, device=DEV)
        flat, g2 = rec.detach(), torch.zeros_like(rec.detach())
        scale = 1.0 / (3.0 * w * h)
        tgt = None if target is None else target[3 * off:3 * (off + w * h)].view(3, h, w).double()
        gv = None if dcolor is None else dcolor[3 * off:3 * (off + w * h)].view(3, h, w)
        for x0, y0, x1, y1, ids in _blocks(rec, ex, ey, key, keep, w, h):
            if ids.numel() == 0:
                continue
            r = flat[:, ids].requires_grad_(want_grad)
            with torch.set_grad_enabled(want_grad):
                cb, tb = _composite64(r, x0, y0, x1, y1)
            cd = cb.detach().view(3, y1 - y0, x1 - x0)
            C[:, y0:y1, x0:x1], T[y0:y1, x0:x1] = cd, tb.detach().view(y1 - y0, x1 - x0)
            if want_grad:
                g = (gv[:, y0:y1, x0:x1] if gv is not None else torch.sign(cd - tgt[:, y0:y1, x0:x1]) * scale)
                (gr,) = torch.autograd.grad(cb, r, g.reshape(3, -1))
                g2.index_add_(1, ids, gr)
        if want_grad:
            (gl,) = torch.autograd.grad(rec, leaf, torch.where(keep, g2, torch.zeros_like(g2)))
            grad += gl
        colors.append(C.reshape(-1))
        Ts.append(T.reshape(-1))
        off += w * h
    out = torch.zeros(planes.shape, dtype=torch.float64, device=DEV)
    out[:, :case["n"]] = grad
    return torch.cat(colors), torch.cat(Ts), out


def _dssim64(x, y, lam):
    """(1 - lam) mean|x - y| + lam (1 - mean SSIM) of (3, h, w) images, and its gradient with respect to x."""
    g = torch.exp(-(torch.arange(11, dtype=torch.float64, device=DEV) - 5) ** 2 / (2 * 1.5 ** 2))
    g = g / g.sum()

    def filt(a):
        a = a[:, None]
        a = torch.nn.functional.conv2d(a, g.view(1, 1, 1, 11), padding=(0, 5))
        return torch.nn.functional.conv2d(a, g.view(1, 1, 11, 1), padding=(5, 0))[:, 0]

    with torch.enable_grad():
        x = x.clone().requires_grad_(True)
        mx, my = filt(x), filt(y)
        sx, sy, sxy = filt(x * x) - mx * mx, filt(y * y) - my * my, filt(x * y) - mx * my
        c1, c2 = 0.01 ** 2, 0.03 ** 2
        s = (2 * mx * my + c1) * (2 * sxy + c2) / ((mx * mx + my * my + c1) * (sx + sy + c2))
        loss = (1 - lam) * (x - y).abs().mean() + lam * (1 - s.mean())
        (gx,) = torch.autograd.grad(loss, x)
    return loss.detach(), gx


def _adam64(case, seed):
    planes, grad, eta, opt = _adam_state(case, seed)
    o, n = opt.opts, case["n"]
    d = lambda v: v[:, :n].double()  # noqa: E731
    p, g, m, v, e = d(planes), d(grad), d(opt.m), d(opt.v), d(eta)
    op, s = torch.sigmoid(p[10]), torch.exp(p[3:6])
    reg = torch.stack([o.lambda_o * op.sum(), o.lambda_sigma * s.sum()])
    g[10] += o.lambda_o * op * (1 - op)
    g[3:6] += o.lambda_sigma * s
    w, x, y, z = p[6:10] / p[6:10].norm(dim=0, keepdim=True)
    R = torch.stack([torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y)]),
                     torch.stack([2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x)]),
                     torch.stack([2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)])])
    tt = torch.einsum("jkn,jn->kn", R, e) * s ** 2
    noise = torch.einsum("jkn,kn->jn", R, tt) * (1 - op) ** (4 * math.exp(o.noise_b)) * (o.lambda_eps * o.lr[0])
    t = opt.t + 1
    m = o.beta1 * m + (1 - o.beta1) * g
    v = o.beta2 * v + (1 - o.beta2) * g * g
    groups = [0] * 3 + [1] * 3 + [2] * 4 + [3, 4] + [5] * 3 + [6, 6, 7, 8, 8, 8] * case["lobes"]
    lr = torch.tensor([o.lr[k] for k in groups], dtype=torch.float64, device=DEV)[:, None]
    p = p - lr * (m / (1 - o.beta1 ** t)) / ((v / (1 - o.beta2 ** t)).sqrt() + o.eps)
    p[0:3] += noise

    def whole(like, new):
        out = like.double()
        out[:, :n] = new
        return out

    return {"planes": whole(planes, p), "m": whole(opt.m, m), "v": whole(opt.v, v), "reg": reg}


def exact(case, seed):
    kind = case["kind"]
    if kind == "adam":
        return _adam64(case, seed)
    if kind == "relocate":
        return None               # picks by the fixed fp32 rule; whole numbers and copies
    if kind == "dssim":
        x, y = _image_pair(case, seed)
        n = 3 * case["width"] * case["height"]
        pairs = [_dssim64(x[k * n:(k + 1) * n].view(3, case["height"], case["width"]).double(),
                          y[k * n:(k + 1) * n].view(3, case["height"], case["width"]).double(), case["ssim"])
                 for k in range(case["views"])]
        return {"loss": torch.stack([a for a, _ in pairs]), "dcolor": torch.cat([b.reshape(-1) for _, b in pairs])}
    grads = kind != "render"
    if _pixels(case) > 2_200_000 or case["n"] > (1_000_000 if grads else 3_200_000):
        return None
    if case["scene"] == "cube" and _pixels(case) * case["n"] > 4e9:
        return None               # thousands of wide primitives on every block
    planes, cams = _scene_planes(case["scene"], case["n"], case["lobes"], seed), _cameras(case)
    if not grads:
        c, t, _ = _render64(planes, case, cams, False)
        return {"color": c, "T": t}
    target = _target(case, seed)
    if kind == "train":
        c, _, _ = _render64(planes, case, cams, False)
        w, h = cams[0].width, cams[0].height
        loss, dl = _dssim64(c.view(3, h, w), target.view(3, h, w).double(), 0.2)
        _, _, g = _render64(planes, case, cams, True, dcolor=dl.reshape(-1))
        return {"color": c, "loss": loss[None], "dcolor": dl.reshape(-1), "grad": g}
    c, _, g = _render64(planes, case, cams, True, target=target)
    views, off = [], 0
    for cam in cams:
        k = 3 * cam.width * cam.height
        views.append((c[off:off + k] - target[off:off + k].double()).abs().mean())
        off += k
    loss = views[0] if kind == "autograd" else torch.stack(views)
    return {"color": c, "loss": loss, "grad": g}
