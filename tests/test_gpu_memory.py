"""Device memory kept between scenes: scenes made and dropped in turn, of changing sizes and on several
threads and streams at once, render what a fresh scene renders (bit-identical), and invalid attributes are
still refused after the one check of all of them."""
from __future__ import annotations

import threading

import numpy as np
import pytest

from paper_2608_15785_gb300 import binding, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_15785_gb300.build import build
    build()


def test_scenes_made_and_dropped_in_turn():
    cam = synth.tiny_camera(160, 120)
    sizes = [300, 9_000, 40_000, 5_000, 1, 70_000, 300]
    scenes = [synth.tiny_scene(n, seed=n) for n in sizes]
    kept = [binding.Scene(sc) for sc in scenes]  # all alive: no memory shared
    want = [[gs.render(cam, mode=m).clone() for m in ("exact", "roofgs")] for gs in kept]
    torch.cuda.synchronize()
    for gs in kept:
        gs.close()
    for _ in range(3):
        for sc, w in zip(scenes, want):
            gs = binding.Scene(sc)
            got = [gs.render(cam, mode=m) for m in ("exact", "roofgs")]
            gs.close()  # with the frames possibly still in flight
            assert all(torch.equal(a, b) for a, b in zip(got, w))


def test_threads_and_streams():
    cam = synth.tiny_camera(160, 120)
    scenes = [synth.tiny_scene(3_000 + 1_000 * k, seed=k) for k in range(4)]
    want = []
    for sc in scenes:
        gs = binding.Scene(sc)
        want.append(gs.render(cam).cpu())
        gs.close()
    errors = []

    def work(k):
        try:
            stream = torch.cuda.Stream()
            for r in range(8):
                j = (k + r) % 4
                with torch.cuda.stream(stream):
                    gs = binding.Scene(scenes[j])
                    img = gs.render(cam)
                    stream.synchronize()
                    if not torch.equal(img.cpu(), want[j]):
                        errors.append((k, r))
                    gs.close()
        except Exception as e:  # reported below: a thread's exception is not the test's
            errors.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors


@pytest.mark.parametrize("storage", [binding.RG_STORE_FP32, binding.RG_STORE_COMPACT])
@pytest.mark.parametrize("field,at,value,text", [
    ("means", (699, 2), np.nan, "non-finite"), ("scales", (0, 0), np.inf, "non-finite"),
    ("quats", (699, 3), -np.inf, "non-finite"), ("sh", (699, 15, 2), np.nan, "non-finite"),
    ("opacities", (699,), np.nan, "non-finite"), ("opacities", (0,), np.float32(1.0000001), "opacity"),
    ("opacities", (350,), -1e-30, "opacity")])
def test_invalid_attributes_are_refused(storage, field, at, value, text):
    sc = synth.tiny_scene(700, seed=2)
    getattr(sc, field)[at] = value
    with pytest.raises(binding.RgError, match=text) as e:
        binding.Scene(sc, storage=storage)
    assert e.value.status == 1


@pytest.mark.parametrize("n,mode", [(5_000, "roofgs"), (40_000, "roofgs"), (40_000, "exact")])
def test_a_reserved_workspace_can_be_captured(n, mode):
    """After a frame and a larger reserve the same view is captured into a graph without an allocation."""
    cam = synth.tiny_camera(320, 240)
    gs = binding.Scene(synth.tiny_scene(n, seed=4))
    want = gs.render(cam, mode=mode).clone()
    gs.reserve(6_000_000)
    out = torch.empty_like(want)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        gs.render(cam, mode=mode, out=out)
    out.zero_()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, want)
    gs.check()


@pytest.mark.parametrize("mode", ["roofgs", "exact"])
@pytest.mark.parametrize("n", [5_000, 40_000])
def test_any_grid_within_the_largest_can_be_captured(n, mode):
    """A view whose tiles are no more than an earlier one's is captured without an allocation, whatever its shape, and so is
    every earlier view after a reserve."""
    wide, tall, small = synth.tiny_camera(960, 64), synth.tiny_camera(64, 960), synth.tiny_camera(160, 120)
    sc = synth.tiny_scene(n, seed=4)
    other = binding.Scene(sc)
    want = [other.render(c, mode=mode).clone() for c in (wide, tall, small)]
    gs = binding.Scene(sc)
    gs.render(wide, mode=mode)

    def captured(cam):
        out = torch.empty((3, cam.height, cam.width), device="cuda")
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            gs.render(cam, mode=mode, out=out)
        g.replay()
        torch.cuda.synchronize()
        return out

    assert torch.equal(captured(tall), want[1])
    gs.render(small, mode=mode)
    gs.reserve(6_000_000)
    for cam, w in zip((wide, tall, small), want):
        assert torch.equal(captured(cam), w)
    gs.check()


def test_trim_gives_the_kept_memory_back():
    """A dropped scene's buffers stay with the library until rg_trim; then other allocators have them, and a new scene is
    made as before."""
    cam = synth.tiny_camera(160, 120)
    sc = synth.tiny_scene(200_000, seed=3)  # 40 MB of SH coefficients
    gs = binding.Scene(sc)
    want = gs.render(cam).clone()
    torch.cuda.synchronize()
    gs.close()
    kept = torch.cuda.mem_get_info()[0]
    binding.trim()
    assert torch.cuda.mem_get_info()[0] - kept >= 30 << 20
    binding.trim()  # nothing left
    assert torch.equal(binding.Scene(sc).render(cam), want)
