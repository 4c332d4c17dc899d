"""The work that a user of this renderer has it do, as cases that can be timed.

A case is a dict of plain values; listed() gives the named ones, draw(rng) more of the same
ranges. prepare() builds what a program holds before the call (a resident scene, a camera, the
output buffer; the frame workspace sized by one checked frame), run() is one pass through the
public entry points, work() what that pass cannot do without, exact() the same outputs in 64
bits from plain torch. The scenes follow the recipes of the package's synthetic workloads
("cube": uniform cube of small Gaussians; "clustered": 20 clusters and a far shell), drawn on
the GPU from the seed; another seed is another scene and another pose.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

from paper_2608_15785_gb300 import binding, synth
from paper_2608_15785_gb300.autograd import render_exact

SHAPES = {"16x16": (16, 16), "32x8": (32, 8), "8x32": (8, 32)}
PIXELS = {1: binding.RG_FLAG_SINGLE_PIXEL, 2: 0, 4: binding.RG_FLAG_QUAD_PIXEL}


def _frame(mode, scene, n, width, height, ppt=2, exp="fast", gauss=False, tile="16x16", bg=0.0):
    """One view through Scene.render: mode, scene recipe and size, image size, pixels per thread,
    exponential, per-Gaussian SH factor, tile shape, background grey level."""
    return {"kind": "frame", "mode": mode, "scene": scene, "n": n, "width": width, "height": height, "ppt": ppt,
            "exp": exp, "gauss": gauss, "tile": tile, "bg": bg}


def listed():
    return [
        # a thumbnail of a small asset: the smallest call, where launches and the host count
        {"name": "roofgs_cube_256", **_frame("roofgs", "cube", 10_000, 256, 256)},
        # a window of odd size in a viewer set for quality: expf, one pixel per thread, wide tiles, a grey backdrop
        {"name": "roofgs_window_quality", **_frame("roofgs", "clustered", 120_000, 1277, 717, ppt=1, exp="exact",
                                                   tile="32x8", bg=0.25)},
        # the everyday viewer frame: 1080p with the defaults
        {"name": "roofgs_1080p", **_frame("roofgs", "clustered", 500_000, 1920, 1080)},
        # the benchmark's frame: 4K, per-Gaussian SH factor, four pixels per thread
        {"name": "roofgs_4k", **_frame("roofgs", "clustered", 3_000_000, 3840, 2160, ppt=4, gauss=True)},
        # a still for a wall or print: 8K
        {"name": "roofgs_8k", **_frame("roofgs", "clustered", 1_000_000, 7680, 4320, ppt=4)},
        # the plain path at a small odd size: a training view scaled down
        {"name": "exact_cube_499x333", **_frame("exact", "cube", 20_000, 499, 333, bg=1.0)},
        # the plain path at 1080p: what RoofGS images are checked against, and a trainer's full view
        {"name": "exact_1080p", **_frame("exact", "clustered", 500_000, 1920, 1080)},
        # the plain path at the benchmark's size
        {"name": "exact_4k", **_frame("exact", "clustered", 3_000_000, 3840, 2160)},
        # the held-out views of a scene rendered together for an image metric: the batched call. Exact
        # mode, whose image does not depend on the pixels per thread that the plan's tuner picks
        {"name": "exact_batch_6_views", "kind": "batch", "n": 150_000, "n2": 40_000, "width": 1280, "height": 720,
         "views": 6},
        # the gradient of a full training view of a resident scene
        {"name": "backward_1080p", "kind": "backward", "scene": "clustered", "n": 500_000, "width": 1920,
         "height": 1080, "tile": "16x16"},
        # one optimisation step's render and gradient through autograd, as a fitting loop calls it
        {"name": "train_step_20k", "kind": "train", "scene": "cube", "n": 20_000, "width": 400, "height": 304},
        # a plugin's sort of its own pairs into depth order, without allocation
        {"name": "sort_pairs_400k", "kind": "sort", "n": 400_000, "bits": 32},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["roofgs", "roofgs", "roofgs", "exact", "exact", "batch", "backward", "train", "sort"])
    if kind == "sort":
        return {"kind": "sort", "n": _log(rng, 1, 524_288), "bits": rng.choice([8, 16, 24, 32])}
    if kind == "train":  # within the first workspace of a fresh scene (2^20 entries)
        return {"kind": "train", "scene": "cube", "n": _log(rng, 500, 40_000), "width": rng.randint(64, 480),
                "height": rng.randint(64, 320)}
    height = _log(rng, 96, 2160)
    width = max(64, min(3840, int(height * rng.choice([1.0, 4 / 3, 16 / 9, 0.6]) + rng.randint(-9, 9))))
    if kind == "batch":
        return {"kind": "batch", "n": _log(rng, 5_000, 300_000), "n2": _log(rng, 2_000, 60_000),
                "width": min(width, 1920), "height": min(height, 1080), "views": rng.randint(1, 8)}
    tile = rng.choice(["16x16", "16x16", "32x8", "8x32"])
    scene = rng.choice(["clustered", "clustered", "cube"])
    n = _log(rng, 2_000, 60_000 if scene == "cube" else 2_000_000)
    if kind == "backward":
        return {"kind": "backward", "scene": scene, "n": min(n, 500_000), "width": min(width, 1920),
                "height": min(height, 1080), "tile": tile}
    if kind == "exact":
        return _frame("exact", scene, n, width, height, tile=tile, bg=rng.choice([0.0, 1.0]))
    return _frame("roofgs", scene, n, width, height, ppt=rng.choice([1, 2, 2, 4, 4]),
                  exp=rng.choice(["fast", "fast", "fast", "exact"]), gauss=rng.random() < 0.5, tile=tile,
                  bg=rng.choice([0.0, 0.5]))


class _Attributes:
    """FP32 attributes of a scene on the GPU, as Scene() takes them."""

    def __init__(self, means, scales, quats, opacities, sh):
        self.means, self.scales, self.quats, self.opacities, self.sh, self.sh_degree = (
            means, scales, quats, opacities, sh, 3)


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _attributes(recipe, n, seed):
    g = _generator(seed)

    def normal(*shape):
        return torch.randn(shape, generator=g, device="cuda")

    def uniform(*shape):
        return torch.rand(shape, generator=g, device="cuda")

    if recipe == "cube":
        means, mu, sigma = uniform(n, 3) * 2 - 1, -4.0, 0.5
    else:
        shell = n // 10
        centres, std = uniform(20, 3) * 3 - 1.5, uniform(20) * 0.35 + 0.05
        weight = -torch.log(uniform(20) + 1e-6)  # normalised exponentials: Dirichlet(1)
        which = torch.multinomial(weight, n - shell, replacement=True, generator=g)
        inner = centres[which] + normal(n - shell, 3) * std[which, None]
        d = torch.nn.functional.normalize(normal(shell, 3), dim=1)
        means = torch.cat([inner, d * (50 * (1 + 0.01 * normal(shell, 1)))])
        mu, sigma = -4.5, 0.8
    sh = normal(n, 16, 3) * 0.3
    sh[:, 0] = sh[:, 0] * (0.2 / 0.3) + 0.5
    return _Attributes(means.contiguous(), torch.exp(mu + sigma * normal(n, 3)),
                       torch.nn.functional.normalize(normal(n, 4), dim=1), torch.sigmoid(1.5 * normal(n)), sh)


def _camera(recipe, width, height, seed, bg=0.0):
    bg = (bg, bg * 0.5, bg)
    if recipe == "cube":
        a = 0.21 * (seed % 30)
        return synth.look_at_camera((3 * math.sin(a), -0.4, -3 * math.cos(a)), width, height, 60.0, 0.2,
                                    3.2 + math.sqrt(3.0), bg=bg)
    return synth.orbit_camera(seed % 30, width, height, bg=bg)


def _batch_cameras(case, seed):
    sizes = [(case["width"], case["height"]), (max(16, case["width"] // 2 + 7), max(16, case["height"] // 2 + 3))]
    return [synth.orbit_camera(seed % 30 + 5 * v, *sizes[v % 2]) for v in range(case["views"])]


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case = case
    kind = case["kind"]
    if kind == "sort":
        g = _generator(seed)
        s.keys0 = torch.randint(-2 ** 31, 2 ** 31, (case["n"],), generator=g, device="cuda", dtype=torch.int32)
        s.vals0 = torch.arange(case["n"], device="cuda", dtype=torch.int32)
        s.keys, s.vals = torch.empty_like(s.keys0), torch.empty_like(s.vals0)
        return s
    if kind == "batch":
        s.scenes = [binding.Scene(_attributes("clustered", case[k], seed + j), storage=binding.RG_STORE_FP32)
                    for j, k in enumerate(("n", "n2"))]
        s.cams = _batch_cameras(case, seed)
        s.which = [v % 2 for v in range(case["views"])]
        # the plan of these views is made by the first call
        s.outs = binding.render_batch(s.scenes, s.which, s.cams, mode="exact", tile=(16, 16))
        return s
    att = _attributes(case["scene"], case["n"], seed)
    s.cam = _camera(case["scene"], case["width"], case["height"], seed, case.get("bg", 0.0))
    shape = (3, case["height"], case["width"])
    if kind == "train":
        s.leaves = {k: getattr(att, k).requires_grad_(True) for k in ("means", "scales", "quats", "opacities", "sh")}
        s.target = torch.rand(shape, generator=_generator(seed + 1), device="cuda")
        return s
    mode = case.get("mode", "exact")
    s.scene = binding.Scene(
        att, storage=binding.RG_STORE_FP32 if mode == "exact" else binding.RG_STORE_COMPACT,
        sh_scale_mode=binding.RG_SH_SCALE_BAND_GAUSS if case.get("gauss") else binding.RG_SH_SCALE_BAND)
    s.tile = SHAPES[case["tile"]]
    s.flags = PIXELS[case.get("ppt", 2)] | (binding.RG_FLAG_EXACT_EXP if case.get("exp") == "exact" else 0)
    s.out = torch.empty(shape, device="cuda")
    # a checked frame sizes the workspace for this view
    s.scene.render(s.cam, mode=mode, flags=s.flags, out=s.out, stats=True, tile=s.tile)
    if kind == "backward":
        s.grad = torch.randn(shape, generator=_generator(seed + 1), device="cuda")
    return s


def run(s):
    kind = s.case["kind"]
    if kind == "frame":
        return s.scene.render(s.cam, mode=s.case["mode"], flags=s.flags, out=s.out, tile=s.tile)
    if kind == "batch":
        return binding.render_batch(s.scenes, s.which, s.cams, mode="exact", outs=s.outs, tile=(16, 16))
    if kind == "backward":
        return s.scene.backward(s.cam, s.grad, tile=s.tile)
    if kind == "train":
        for t in s.leaves.values():
            t.grad = None
        img = render_exact(*s.leaves.values(), s.cam)
        loss = ((img - s.target) ** 2).mean()
        loss.backward()
        return {"image": img.detach(), "loss": loss.detach(), **{k: t.grad for k, t in s.leaves.items()}}
    s.keys.copy_(s.keys0)  # the sort works in place; a caller's arrays are fresh each time
    s.vals.copy_(s.vals0)
    binding.check(binding.lib().rg_sort_pairs_noalloc(
        ctypes.c_void_p(s.keys.data_ptr()), ctypes.c_void_p(s.vals.data_ptr()), s.case["n"], s.case["bits"], None,
        ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)))
    return s.keys, s.vals


def work(case):
    """Scene read once, images (and gradients) written once; the operations of about 400 per
    Gaussian (projection, covariance, SH) and of about 60 blended pairs a pixel at 20 each, the
    depth at which the opacities of these scenes saturate a pixel."""
    kind = case["kind"]
    if kind == "sort":
        return {"bytes": 16.0 * case["n"], "flops": 0.0}
    if kind == "batch":
        cams = _batch_cameras(case, 0)
        px = sum(c.width * c.height for c in cams)
        n = sum(case["n"] if v % 2 == 0 else case["n2"] for v in range(case["views"]))
        return {"bytes": 236.0 * n + 12.0 * px, "flops": 400.0 * n + 1200.0 * px}
    n, px = case["n"], case["width"] * case["height"]
    if kind == "frame":
        per = 236.0 if case["mode"] == "exact" else 80.0
        return {"bytes": per * n + 12.0 * px, "flops": 400.0 * n + 1200.0 * px}
    # forward image (train only), dL/dimage, attributes in, gradients out
    images = 24.0 if kind == "train" else 12.0
    return {"bytes": 472.0 * n + images * px, "flops": 1500.0 * n + 4800.0 * px}


# ---------------------------------------------------------------------------------------------
# The same outputs in 64 bits. Whole-number decisions (culling, tile rectangles, quantised depth,
# the INT8 / FP16 storage of the compact attributes) are FP32 by definition and are taken in FP32;
# every value that reaches a pixel is computed in 64 bits.
# ---------------------------------------------------------------------------------------------
LN255 = float(np.float32(5.541263545158426))


def _f32(x):
    return torch.tensor(x, dtype=torch.float32, device="cuda")


def _dot3(m, r, t=None):
    s = (r[0] * m[:, 0] + r[1] * m[:, 1]) + r[2] * m[:, 2]
    return s if t is None else s + t


def _rotation(q):
    n = torch.sqrt(((q[:, 0] * q[:, 0] + q[:, 1] * q[:, 1]) + q[:, 2] * q[:, 2]) + q[:, 3] * q[:, 3])
    w, x, y, z = (q[:, k] / n for k in range(4))
    return [1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
            2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
            2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)]


def _project(means, scales, quats, cam, dtype):
    """Projected mean, Sigma' and its determinant, camera depth, in `dtype`."""
    R = torch.as_tensor(np.asarray(cam.R, np.float32), device="cuda").to(dtype)
    t = torch.as_tensor(np.asarray(cam.t, np.float32), device="cuda").to(dtype)
    fx, fy, cx, cy = (_f32(v).to(dtype) for v in (cam.fx, cam.fy, cam.cx, cam.cy))
    px, py, pz = (_dot3(means, R[3 * k:3 * k + 3], t[k]) for k in range(3))
    Q = _rotation(quats)
    M = [Q[3 * i + k] * scales[:, k] for i in range(3) for k in range(3)]
    xz, yz = px / pz, py / pz
    limx = (_f32(1.3) * ((_f32(0.5) * _f32(float(cam.width))) / _f32(cam.fx))).to(dtype)
    limy = (_f32(1.3) * ((_f32(0.5) * _f32(float(cam.height))) / _f32(cam.fy))).to(dtype)
    cxz, cyz = torch.minimum(limx, torch.maximum(-limx, xz)), torch.minimum(limy, torch.maximum(-limy, yz))
    j00, j11 = fx / pz, fy / pz
    j02, j12 = -(j00 * cxz), -(j11 * cyz)
    A = [j00 * R[k] + j02 * R[6 + k] for k in range(3)] + [j11 * R[3 + k] + j12 * R[6 + k] for k in range(3)]
    U = [(A[3 * i] * M[k] + A[3 * i + 1] * M[3 + k]) + A[3 * i + 2] * M[6 + k] for i in range(2) for k in range(3)]
    n0 = (U[0] * U[0] + U[1] * U[1]) + U[2] * U[2]
    n1 = (U[3] * U[3] + U[4] * U[4]) + U[5] * U[5]
    dil = _f32(0.3).to(dtype)
    sa, sc = n0 + dil, n1 + dil
    sb = (U[0] * U[3] + U[1] * U[4]) + U[2] * U[5]
    c0, c1, c2 = U[1] * U[5] - U[2] * U[4], U[2] * U[3] - U[0] * U[5], U[0] * U[4] - U[1] * U[3]
    det = (((c0 * c0 + c1 * c1) + c2 * c2) + dil * (n0 + n1)) + _f32(0.09).to(dtype)
    return fx * xz + cx, fy * yz + cy, sa, sb, sc, det, pz


def _basis(d):
    x, y, z = d[:, 0], d[:, 1], d[:, 2]
    k1, k2, k3 = math.sqrt(3 / (4 * math.pi)), math.sqrt(15 / (4 * math.pi)), math.sqrt(35 / (32 * math.pi))
    a, b = math.sqrt(105 / (4 * math.pi)), math.sqrt(21 / (32 * math.pi))
    return torch.stack([
        torch.full_like(x, math.sqrt(1 / (4 * math.pi))), k1 * y, k1 * z, k1 * x, k2 * x * y, k2 * y * z,
        math.sqrt(5 / (16 * math.pi)) * (3 * z * z - 1), k2 * x * z, 0.5 * k2 * (x * x - y * y),
        k3 * y * (3 * x * x - y * y), a * x * y * z, b * y * (5 * z * z - 1),
        math.sqrt(7 / (16 * math.pi)) * z * (5 * z * z - 3), b * x * (5 * z * z - 1), 0.5 * a * z * (x * x - y * y),
        k3 * x * (x * x - 3 * y * y)], 1)


def _colour(means, sh, cam):
    R, t = (torch.as_tensor(np.asarray(v, np.float64), device="cuda") for v in (cam.R, cam.t))
    v = means + R.reshape(3, 3).T @ t
    Y = _basis(v / torch.sqrt((v * v).sum(1, keepdim=True)))
    return torch.clamp((Y[:, :, None] * sh).sum(1) + 0.5, 0, 1)


def _compact(att, gauss):
    """The stored values of the compact attributes as FP32 tensors: FP16 geometry, SH codes times scales."""
    sh = att.sh
    band = torch.tensor([0] + [1] * 3 + [2] * 5 + [3] * 7, device="cuda")
    top = torch.zeros(4, 3, device="cuda")
    for b in range(4):
        top[b] = sh[:, band == b].abs().amax(dim=(0, 1))
    scale = (top / 127.0)[band]  # [16, 3]
    if gauss:
        g = (sh.abs() / (127.0 * scale)).amax(dim=(1, 2)).half().float()[:, None, None]
        den = g * scale
    else:
        g, den = torch.ones(sh.shape[0], 1, 1, device="cuda"), scale.expand_as(sh)
    code = torch.clamp(torch.round(sh / den), -127, 127)
    return att.quats.half().float(), att.scales.half().float(), code.double() * scale.double() * g.double()


def _entries(cam, tile, u, v, sa, sb, sc, det, front, tt):
    """(Gaussian, tile) pairs in Gaussian order; tt None: the 3-sigma box, else the 1/255 ellipse per tile row."""
    tw, th = tile
    if tt is None:
        h = 0.5 * (sa - sc)
        rx = ry = torch.ceil(3.0 * torch.sqrt(0.5 * (sa + sc) + torch.sqrt(h * h + sb * sb)))
    else:
        rx, ry = torch.sqrt(tt * sa), torch.sqrt(tt * sc)
    xl, xh = torch.ceil(u - rx).clamp(min=0), torch.floor(u + rx).clamp(max=cam.width - 1)
    yl, yh = torch.ceil(v - ry).clamp(min=0), torch.floor(v + ry).clamp(max=cam.height - 1)
    ok = front & torch.isfinite(u) & torch.isfinite(v) & torch.isfinite(rx) & torch.isfinite(ry) & (xl <= xh) & (yl <= yh)
    gid = torch.nonzero(ok).squeeze(1)
    ty0, ty1 = yl[gid].long() // th, yh[gid].long() // th
    rows = ty1 - ty0 + 1
    rg = torch.repeat_interleave(torch.arange(gid.numel(), device="cuda"), rows)
    ty = ty0[rg] + (torch.arange(rg.numel(), device="cuda") - (rows.cumsum(0) - rows)[rg])
    i = gid[rg]
    if tt is None:
        a0, a1 = xl[i], xh[i]
    else:
        ys = sb * torch.sqrt(tt / sa)
        cc, kk, isc = sb / sc, torch.sqrt(det / sc), 1.0 / sc
        d0 = torch.maximum((ty * th).float(), yl[i]) - v[i]
        d1 = torch.minimum((ty * th + th - 1).float(), yh[i]) - v[i]
        dmax = torch.minimum(torch.maximum(ys[i], d0), d1)
        dmin = torch.minimum(torch.maximum(-ys[i], d0), d1)
        wr = torch.sqrt((tt[i] - (dmax * dmax) * isc[i]).clamp(min=0))
        wl = torch.sqrt((tt[i] - (dmin * dmin) * isc[i]).clamp(min=0))
        xr = (u[i] + cc[i] * dmax) + kk[i] * wr
        xf = (u[i] + cc[i] * dmin) - kk[i] * wl
        a0, a1 = torch.maximum(torch.ceil(xf), xl[i]), torch.minimum(torch.floor(xr), xh[i])
    keep = a0 <= a1
    i, ty, t0, t1 = i[keep], ty[keep], a0[keep].long() // tw, a1[keep].long() // tw
    w = t1 - t0 + 1
    e = torch.repeat_interleave(torch.arange(w.numel(), device="cuda"), w)
    tx = t0[e] + (torch.arange(e.numel(), device="cuda") - (w.cumsum(0) - w)[e])
    return i[e], ty[e] * ((cam.width + tw - 1) // tw) + tx


class _Blend:
    """Front-to-back blend over the sorted tile lists in 64 bits, 2048 tiles and 16 pairs at a time;
    with `grad`, the gradient with respect to the per-Gaussian (u, v, A, B, C, o, rgb) as well."""

    TILES, PAIRS = 2048, 16

    def __init__(self, cam, tile, gauss, tiles, order, params, kind):
        tw, th = tile
        self.cam, self.kind, self.p = cam, kind, params
        self.nx = (cam.width + tw - 1) // tw
        self.count = self.nx * ((cam.height + th - 1) // th)
        rank = torch.empty_like(order)
        rank[order] = torch.arange(order.numel(), device="cuda")
        key = torch.sort(tiles * max(1, order.numel()) + rank[gauss])[0]
        self.g = order[key % max(1, order.numel())]
        self.len = torch.bincount(tiles, minlength=self.count)
        self.start = self.len.cumsum(0) - self.len
        k = torch.arange(tw * th, device="cuda")
        self.lx, self.ly, self.tw, self.th = k % tw, k // tw, tw, th

    def step(self, q, valid, x, y, T):
        """16 pairs: q [A, K, 9]; new transmittance, colour added, and whether the pixel ended."""
        dx, dy = x[:, None] - q[..., 0, None], y[:, None] - q[..., 1, None]
        p = -0.5 * (q[..., 2, None] * dx * dx + q[..., 4, None] * dy * dy) - q[..., 3, None] * dx * dy
        if self.kind == "plain":
            a = torch.clamp(q[..., 5, None] * torch.exp(p), max=0.99)
            use = a >= 1.0 / 255.0
        else:
            p = p + q[..., 5, None]
            use = p >= -LN255
            if self.kind == "exact":
                a = torch.exp(p)
            else:
                w = p.clamp(min=-LN255) * float(np.float32(1.44269502)) + float(np.float32(126.954323))
                a = torch.ldexp(1.0 + (w - torch.floor(w)), torch.floor(w) - 127.0)
            a = torch.clamp(a, max=0.99)
        a = torch.where(use & valid[..., None], a, torch.zeros_like(a))
        after = T[:, None] * torch.cumprod(1 - a, 1)
        live = after.detach() >= 1e-4
        a = torch.where(live, a, torch.zeros_like(a))
        after = T[:, None] * torch.cumprod(1 - a, 1)
        before = torch.cat([T[:, None], after[:, :-1]], 1)
        return after[:, -1], torch.einsum("akp,akc->apc", a * before, q[..., 6:9]), ~live[:, -1]

    def group(self, t, upto):
        """The steps of the tiles t: (their rows, Gaussians, validity) of each 16 pairs."""
        for k in range(0, upto, self.PAIRS):
            j = k + torch.arange(self.PAIRS, device="cuda")
            valid = j[None] < self.len[t][:, None]
            yield k, self.g[(self.start[t][:, None] + j[None]).clamp(max=max(0, self.g.numel() - 1))], valid

    def __call__(self, grad=None):
        W, H = self.cam.width, self.cam.height
        bg = torch.as_tensor(np.asarray(self.cam.bg, np.float32), device="cuda").double()
        img = torch.zeros(3, H, W, dtype=torch.float64, device="cuda")
        dp = torch.zeros_like(self.p) if grad is not None else None
        todo = torch.argsort(self.len, descending=True)
        for b in range(0, self.count, self.TILES):
            t = todo[b:b + self.TILES]
            x = (t % self.nx * self.tw)[:, None] + self.lx
            y = (t // self.nx * self.th)[:, None] + self.ly
            inside = (x < W) & (y < H)
            T = torch.ones(x.shape, dtype=torch.float64, device="cuda")
            C = torch.zeros(*x.shape, 3, dtype=torch.float64, device="cuda")
            done, tape = ~inside, []
            if self.g.numel():
                for _, g, valid in self.group(t, int(self.len[t[0]])):
                    if bool(done.all()):
                        break
                    Tn, add, end = self.step(self.p[g], valid, x, y, T)
                    if grad is not None:
                        tape.append((g, valid, T, done))
                    C = torch.where(done[..., None], C, C + add)
                    T = torch.where(done, T, Tn)
                    done = done | end
            full = C + T[..., None] * bg
            img[:, y[inside], x[inside]] = full[inside].T
            if grad is None:
                continue
            G = torch.zeros_like(C)
            G[inside] = grad[:, y[inside], x[inside]].T
            dT = (G * bg).sum(-1)
            for g, valid, T, done in reversed(tape):
                with torch.enable_grad():
                    q = self.p[g].requires_grad_(True)
                    Ti = T.clone().requires_grad_(True)
                    Tn, add, _ = self.step(q, valid, x, y, Ti)
                    live = (~done).double()
                    out = (Tn * dT * live).sum() + (add * G * live[..., None]).sum()
                    dq, dTi = torch.autograd.grad(out, (q, Ti))
                dT = torch.where(done, dT, dTi)
                dp.index_add_(0, g.reshape(-1), dq.reshape(-1, 9))
        return img, dp


def _reference(att, cam, tile, mode, exp, gauss, grad=None):
    """Image (and, for a dL/dimage or a function of the image that gives it, the gradients) in 64 bits."""
    if mode == "roofgs":
        quats, scales, sh = _compact(att, gauss)
        logo = torch.log(att.opacities.double()).float()
    else:
        quats, scales, sh, logo = att.quats, att.scales, att.sh.double(), None
    u, v, sa, sb, sc, det, pz = _project(att.means, scales, quats, cam, torch.float32)
    zn, zf = _f32(cam.znear), _f32(cam.zfar)
    front = (pz > zn) & (pz <= zf)
    nx, ny = -(-cam.width // tile[0]), -(-cam.height // tile[1])
    if mode == "roofgs":
        front = front & (logo >= -LN255)
        tt = 2.0 * (logo + _f32(LN255))
        bd = 32 - (nx * ny - 1).bit_length()
        qmax = float(2 ** bd - 1)
        scale = _f32(float(np.float32(qmax / (float(np.float32(cam.zfar)) - float(np.float32(cam.znear))))))
        order = torch.argsort(torch.floor((pz - zn) * scale).clamp(0, qmax).double(), stable=True)
    else:
        tt = None
        order = torch.argsort(pz, stable=True)
    gauss_id, tiles = _entries(cam, tile, u, v, sa, sb, sc, det, front, tt)
    leaves = [x.double().requires_grad_(grad is not None)
              for x in (att.means, scales, quats, att.opacities if logo is None else logo, sh)]
    with torch.set_grad_enabled(grad is not None):
        u, v, sa, sb, sc, det, _ = _project(leaves[0], leaves[1], leaves[2], cam, torch.float64)
        params = torch.cat([torch.stack([u, v, sc / det, -sb / det, sa / det, leaves[3]], 1),
                            _colour(leaves[0], leaves[4], cam)], 1)
    kind = "plain" if mode == "exact" else exp
    blend = _Blend(cam, tile, gauss_id, tiles, order, params.detach(), kind)
    if grad is None:
        return blend()[0], None
    g = grad(blend()[0]) if callable(grad) else grad
    img, dp = blend(g)
    seen = torch.zeros(att.means.shape[0], 1, dtype=torch.bool, device="cuda")
    seen[gauss_id] = True
    dp = torch.where(seen, dp, torch.zeros_like(dp))
    safe = torch.where(seen, params, params.detach())
    got = torch.autograd.grad((safe * dp).sum(), leaves)
    got = [torch.where(seen.reshape(-1, *[1] * (x.dim() - 1)), x, torch.zeros_like(x)) for x in got]
    return img, dict(zip(("means", "scales", "quats", "opacities", "sh"), got))


def exact(case, seed):
    kind = case["kind"]
    if kind == "sort":
        return None  # whole numbers
    if kind == "batch":
        att = [_attributes("clustered", case[k], seed + j) for j, k in enumerate(("n", "n2"))]
        return [_reference(att[v % 2], c, (16, 16), "exact", "exact", False)[0]
                for v, c in enumerate(_batch_cameras(case, seed))]
    if kind == "frame" and case["width"] * case["height"] > 12_000_000:
        return None  # over 20 seconds
    att = _attributes(case["scene"], case["n"], seed)
    cam = _camera(case["scene"], case["width"], case["height"], seed, case.get("bg", 0.0))
    if kind == "frame":
        return _reference(att, cam, SHAPES[case["tile"]], case["mode"], case["exp"], case["gauss"])[0]
    shape = (3, case["height"], case["width"])
    if kind == "backward":
        grad = torch.randn(shape, generator=_generator(seed + 1), device="cuda").double()
        return _reference(att, cam, SHAPES[case["tile"]], "exact", "exact", False, grad)[1]
    target = torch.rand(shape, generator=_generator(seed + 1), device="cuda").double()
    img, got = _reference(att, cam, (16, 16), "exact", "exact", False, lambda im: 2 * (im - target) / im.numel())
    return {"image": img, "loss": ((img - target) ** 2).mean(), **got}
