"""Backward of the exact-mode render (rg_backward), through the C ABI.

Reference: central finite differences of the FP64 oracle render of
L = sum(w * image) with fixed random weights w, on a 256x256 view of a
1,000-Gaussian subset. The forward is piecewise smooth (the 1/255 skip, the
1e-4 stop and the 0.99 clamp are kinks or steps), so every finite difference is
taken with two step sizes and a sample whose two estimates disagree (it sits
on a step) is set aside and counted; the rest must match the GPU gradient.
"""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_2608_15785_gb300 import binding, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_15785_gb300.build import build
    build()


def _scene():
    full = synth.tiny_scene(10_000, seed=0)
    rng = np.random.default_rng(4)
    idx = np.sort(rng.choice(full.n, 1000, replace=False))
    sc = full.subset(idx)
    sc.scales = (sc.scales * 2.5).astype(np.float32)  # fewer, larger Gaussians: more pixels per gradient
    return sc


def _loss_oracle(sc, cam, w):
    img, _, _ = oracle.render(sc, cam, oracle.EXACT, with_diag=False)
    return float(np.sum(w * img))


FIELDS = {"means": 3, "scales": 3, "quats": 4, "opacities": 1, "sh": 48}


def _perturbed(sc, field, i, k, value):
    out = sc.subset(np.arange(sc.n))
    arr = getattr(out, field)
    if field == "sh":
        arr[i].reshape(-1)[k] = value
    elif arr.ndim == 1:
        arr[i] = value
    else:
        arr[i, k] = value
    return out


def _get(sc, field, i, k):
    arr = getattr(sc, field)
    if field == "sh":
        return float(arr[i].reshape(-1)[k])
    return float(arr[i] if arr.ndim == 1 else arr[i, k])


def _fd(sc, cam, w, field, i, k, rel):
    x0 = _get(sc, field, i, k)
    h = rel * max(abs(x0), 0.05 if field != "sh" else 0.3)
    xp, xm = np.float32(x0 + h), np.float32(x0 - h)
    lp = _loss_oracle(_perturbed(sc, field, i, k, xp), cam, w)
    lm = _loss_oracle(_perturbed(sc, field, i, k, xm), cam, w)
    return (lp - lm) / (float(xp) - float(xm))


def test_backward_matches_fp64_finite_differences():
    sc = _scene()
    cam = synth.tiny_camera(256, 256, bg=(0.1, 0.3, 0.2))
    rng = np.random.default_rng(7)
    w = rng.normal(size=(3, 256, 256))
    gs = binding.Scene(sc, storage=binding.RG_STORE_FP32)
    g = gs.backward(cam, torch.from_numpy(w.astype(np.float32)).cuda())
    torch.cuda.synchronize()
    g = {k: v.cpu().numpy().astype(np.float64) for k, v in g.items()}
    # Gaussians that reach the image
    k_, v_, _, _ = oracle.keys(sc, cam, oracle.EXACT)
    vis = np.unique(v_)
    samples = []
    for field, dim in FIELDS.items():
        for _ in range(8 if field != "sh" else 10):
            i = int(rng.choice(vis))
            k = int(rng.integers(dim))
            if field == "sh":
                k = int(rng.integers(3)) if _ < 4 else k  # include DC terms
            samples.append((field, i, k))
    checked = skipped = 0
    scale = {f: np.abs(g[f][vis]).mean() + 1e-12 for f in FIELDS}
    for field, i, k in samples:
        a = _fd(sc, cam, w, field, i, k, 1e-4)
        b = _fd(sc, cam, w, field, i, k, 5e-5)
        if abs(a - b) > 1e-3 * (abs(a) + scale[field]):
            skipped += 1  # a skip/stop/clamp step lies within the difference interval
            continue
        gv = g[field][i].reshape(-1)[k] if field == "sh" else (g[field][i] if g[field].ndim == 1 else g[field][i, k])
        assert abs(gv - a) <= 2e-3 * abs(a) + 2e-3 * scale[field], (field, i, k, gv, a)
        checked += 1
    print("backward: %d gradients checked against FP64 finite differences, %d on a step set aside" %
          (checked, skipped))
    assert checked >= 0.8 * len(samples)


def test_backward_matches_fp32_gpu_finite_differences():
    """Coarse second reference: central differences of the GPU forward itself."""
    sc = _scene()
    cam = synth.tiny_camera(256, 256)
    rng = np.random.default_rng(9)
    w = torch.from_numpy(rng.normal(size=(3, 256, 256)).astype(np.float32)).cuda()
    g = binding.Scene(sc, storage=binding.RG_STORE_FP32).backward(cam, w)
    gm = g["means"].cpu().numpy()
    top = np.argsort(-np.abs(gm[:, 0]))[:8]  # the largest x-gradients are well above FP32 noise

    def fd(i, h):
        vals = []
        for sgn in (+1, -1):
            s2 = sc.subset(np.arange(sc.n))
            s2.means[i, 0] = np.float32(s2.means[i, 0] + sgn * h)
            img = binding.Scene(s2, storage=binding.RG_STORE_FP32).render(cam, mode="exact")
            vals.append(float((img.double() * w.double()).sum()))
        return (vals[0] - vals[1]) / (2 * h)

    checked = 0
    for i in top:
        a, b = fd(i, 1e-3), fd(i, 5e-4)
        if abs(a - b) > 0.02 * abs(a):
            continue  # a step of the forward lies within the interval
        assert abs(a - gm[i, 0]) <= 0.05 * abs(gm[i, 0]), (i, a, gm[i, 0])
        checked += 1
    assert checked >= 4


def test_autograd_function_and_unsupported_mode():
    from paper_2608_15785_gb300.autograd import render_exact
    sc = _scene()
    cam = synth.tiny_camera(128, 96)
    t = {f: torch.from_numpy(getattr(sc, f)).cuda().requires_grad_(True)
         for f in ("means", "scales", "quats", "opacities", "sh")}
    w = torch.randn(3, 96, 128, device="cuda")
    img = render_exact(t["means"], t["scales"], t["quats"], t["opacities"], t["sh"], cam)
    (img * w).sum().backward()
    ref = binding.Scene(sc, storage=binding.RG_STORE_FP32).backward(cam, w)
    for f in t:
        # the per-Gaussian sums use atomics, so two backward runs agree to rounding only
        assert torch.allclose(t[f].grad, ref[f], rtol=1e-4, atol=1e-5 * float(ref[f].abs().max())), f
    gs = binding.Scene(sc)
    import ctypes as C
    o = binding.RgOpts(binding.RG_MODE_ROOFGS, 0, 16, 16)
    c = binding.camera_struct(cam)
    gg = binding.RgGrads(*(ref[k].data_ptr() for k in ("means", "scales", "quats", "opacities", "sh")))
    assert binding.lib().rg_backward(gs.handle, C.byref(c), C.byref(o), C.c_void_p(w.data_ptr()), C.byref(gg),
                                     None) == 8


def test_backward_matches_fp64_oracle_gradient_everywhere():
    """rg_backward against the oracle's FP64 analytic gradient (oracle.backward), element by
    element over every Gaussian of the 1,000-Gaussian 256x256 crop and every attribute.
    Tolerance per attribute kind: |GPU - FP64| <= 2e-3 |FP64| + 2e-4 * max|FP64| (the
    GPU sums FP32 per-pixel terms with atomics and runs the chain rule in FP32)."""
    sc = _scene()
    cam = synth.tiny_camera(256, 256, bg=(0.1, 0.3, 0.2))
    w = np.random.default_rng(11).normal(size=(3, 256, 256))
    g = binding.Scene(sc, storage=binding.RG_STORE_FP32).backward(cam, torch.from_numpy(w.astype(np.float32)).cuda())
    torch.cuda.synchronize()
    ref = oracle.backward(sc, cam, w.astype(np.float32).astype(np.float64))
    for f in FIELDS:
        a = g[f].cpu().numpy().astype(np.float64).reshape(sc.n, -1)
        b = ref[f].reshape(sc.n, -1)
        scale = float(np.abs(b).max())
        err = np.abs(a - b)
        rel = err / (np.abs(b) + 1e-300)
        print("backward %s: max |err| %.3g (max |g| %.3g), median rel %.2g, 99th pct rel %.2g" % (
            f, float(err.max()), scale, float(np.median(rel[np.abs(b) > 1e-3 * scale])),
            float(np.percentile(rel[np.abs(b) > 1e-3 * scale], 99))))
        bad = err > 2e-4 * np.abs(b) + 2e-5 * scale
        assert not bad.any(), (f, int(bad.sum()), np.argwhere(bad)[:5].tolist())


def _cancelling_camera(width, height):
    """z of the mean (2^24 + 2, 1, 3) is 2 in FP32 and 0 exactly, so its projected mean is no number."""
    R = np.array([0, 1, 0, 0, 0, 1, 1, 1, 1], np.float32)
    t = np.array([-1.0, -3.0, -(2.0 ** 24 + 6.0)], np.float32)
    return synth.Camera(R, t, 100.0, 100.0, (width - 1) / 2.0, (height - 1) / 2.0, width, height, 0.5, 100.0)


def _undefined_scene(opacity):
    """That Gaussian, its rectangle about 30 pixels wide, in front of an ordinary one as wide."""
    sc = synth.tiny_scene(2, seed=1)
    sc.means = np.array([[2 ** 24 + 2, 1, 3], [2 ** 24 + 40, 1, 3]], np.float32)
    sc.scales = np.array([[0.1] * 3, [2.0] * 3], np.float32)
    sc.opacities = np.array([opacity, 0.7], np.float32)
    return sc


# two and four pixels per thread
@pytest.mark.parametrize("wh", [(160, 120), (1024, 1040)])
@pytest.mark.parametrize("opacity", [0.0, 0.5, 1.0])
def test_a_gaussian_without_an_exponent(wh, opacity):
    """alpha = min(0.99, o expf(NaN)) = 0.99: the timed image equals the counting launch's, which has the Gaussian all over
    its rectangle, and the gradients are of that image: what lies behind gets 1 - 0.99 of its own (to rounding: 1e-4), the
    Gaussian itself a number for its colour alone."""
    cam = _cancelling_camera(*wh)
    sc = _undefined_scene(opacity)
    gs = binding.Scene(sc, storage=binding.RG_STORE_FP32)
    img = gs.render(cam, mode="exact").clone()
    full, st = gs.render(cam, mode="exact", stats=True)
    assert st["n_visible"] == 2
    behind = binding.Scene(sc.subset([1]), storage=binding.RG_STORE_FP32)
    alone = behind.render(cam, mode="exact")
    inside = (full != alone).any(0)
    assert int(inside.sum()) >= 256
    assert torch.equal(img, full)
    w = torch.randn((3, wh[1], wh[0]), generator=torch.Generator().manual_seed(5)).cuda() * inside
    g, ref = gs.backward(cam, w), behind.backward(cam, w)
    left = float(np.float32(1) - np.float32(0.99))
    for f in ref:
        b = ref[f][0] * left
        if f != "quats":  # (zero for equal scales: rounding alone)
            assert torch.allclose(g[f][1], b, rtol=1e-4, atol=1e-4 * float(b.abs().max())), f
        if f == "sh":
            assert bool(torch.isfinite(g[f][0]).all()) and bool((g[f][0] != 0).any())
        else:
            assert bool(torch.isnan(g[f][0]).all()), f


# two and four pixels per thread; a pixel of each half of a pair
@pytest.mark.parametrize("wh", [(256, 192), (1024, 1040)])
@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan, 3e38])
def test_a_non_finite_gradient_stays_with_its_pixel(wh, value):
    """A Gaussian that the pixel does not blend (alpha < 1/255 there by a wide margin, or culled) has the gradients that a
    zero in the pixel's place gives it, to rounding (the sums use atomics); the first one that it surely blends has no number."""
    rng = np.random.default_rng(3)
    sc = synth.tiny_scene(600, seed=8)
    sc.scales = (sc.scales * 2.0).astype(np.float32)
    cam = synth.tiny_camera(*wh, bg=(0.1, 0.3, 0.2))
    # specks about the two pixels, many of which reach only the neighbours that share a thread
    sc.means[:200] = np.append(rng.uniform(-5, 10, (200, 2)) / cam.fx * 3.0, rng.uniform(-0.01, 0.01, (200, 1)), 1)
    sc.scales[:200] = np.float32(1.0 / cam.fx)
    sc.opacities[:200] = 0.1
    gs = binding.Scene(sc, storage=binding.RG_STORE_FP32)
    w = torch.from_numpy(rng.normal(size=(3, wh[1], wh[0])).astype(np.float32)).cuda()
    far = np.zeros(sc.n, bool)
    for x, y in ((wh[0] // 2, wh[1] // 2), (wh[0] // 2 + 5, wh[1] // 2 + 1)):
        d2, z = np.empty(sc.n), np.empty(sc.n)
        for i in range(sc.n):
            p = oracle.project64(sc.means[i], sc.quats[i], sc.scales[i], cam)
            d = np.array([p["u"] - x, p["v"] - y])
            d2[i], z[i] = d @ np.linalg.solve(p["cov2d"], d), p["z"]
        power = np.log(np.maximum(sc.opacities, 1e-30)) - 0.5 * d2
        far = power < np.log(0.5 / 255.0)
        front = int(np.argmin(np.where((power > np.log(0.05)) & (sc.opacities < 0.98), z, np.inf)))
        zero, bad = w.clone(), w.clone()
        zero[1, y, x] = 0.0
        bad[1, y, x] = float(value)
        ref, g = gs.backward(cam, zero), gs.backward(cam, bad)
        keep = torch.from_numpy(far).cuda()
        assert 100 < int(keep.sum()) < sc.n
        for f in FIELDS:
            assert torch.allclose(g[f][keep], ref[f][keep], rtol=1e-4, atol=1e-5 * float(ref[f].abs().max())), f
        assert np.isfinite(value) or not bool(torch.isfinite(g["opacities"][front]))
