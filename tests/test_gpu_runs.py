"""Entries written from tile-row runs (the default RoofGS frame) at the sizes where their grouping
changes shape: entries, ranges, counters and images bit-identical to the fused front end's with its
radix passes, whose own parity with the oracle is tested elsewhere. Whole numbers: exact equality."""
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


def _entries(gs):
    return [gs.inspect(k) for k in (binding.RG_INSPECT_KEYS, binding.RG_INSPECT_VALUES, binding.RG_INSPECT_RANGES)]


def _scene(n, scale=1.0, seed=3):
    sc = synth.tiny_scene(n, seed=seed)
    sc.scales = (sc.scales * np.float32(scale)).astype(np.float32)
    return sc


# n around the last small frame (128 blocks of 256 Gaussians); few tile rows with many runs each (several
# chunks per row); sparse rows over more than 1,024 front-end blocks; 512 tile columns and rows (the
# largest grid of runs, column groups) and 513 (the fused front end); one tile
CASES = [(255, (64, 48), (16, 16), 1.0), (32_768, (256, 256), (16, 16), 1.0), (32_769, (256, 256), (16, 16), 1.0),
         (60_000, (90, 40), (16, 16), 1.0), (400_000, (48, 48), (8, 32), 0.5), (300_000, (640, 1600), (32, 8), 0.05),
         (4_000, (8192, 40), (16, 16), 3.0), (4_000, (40, 8192), (16, 16), 3.0), (40_000, (8192, 40), (16, 16), 2.0),
         (4_000, (8208, 40), (16, 16), 3.0), (4_000, (40, 8208), (16, 16), 3.0), (5_000, (5, 7), (16, 16), 4.0)]


@pytest.mark.parametrize("n,wh,tile,scale", CASES)
def test_runs_equal_the_ordered_front_end(n, wh, tile, scale):
    cam = synth.tiny_camera(*wh, bg=(0.2, 0.1, 0.3))
    if wh[1] > 4 * wh[0]:
        cam.fx = cam.fy = float(np.float32(wh[1] * 0.8))  # the cube over the whole height
    gs = binding.Scene(_scene(n, scale))
    a, sa = gs.render(cam, flags=binding.RG_FLAG_QUAD_PIXEL, stats=True, tile=tile)
    ea = _entries(gs)
    # (the first image is the counting launch's)
    a = gs.render(cam, flags=binding.RG_FLAG_QUAD_PIXEL, tile=tile)
    b, sb = gs.render(cam, flags=binding.RG_FLAG_QUAD_PIXEL | binding.RG_FLAG_ORDERED_FRONT_END, stats=True, tile=tile)
    eb = _entries(gs)
    assert sa["n_entries"] > 0
    for f in ("n_entries", "n_visible", "n_front", "n_pairs", "n_blends"):
        assert sa[f] == sb[f], f
    for x, y in zip(ea, eb):
        assert np.array_equal(x, y)
    assert torch.equal(a, b)
    gs.check()


@pytest.mark.parametrize("n", [20_000, 40_000])
def test_runs_beyond_the_capacity(n):
    """A small and a larger frame with too few entries of room: the kept entries are those whose place
    in (tile row, depth code, index, tile column) order lies below the capacity; the re-rendered frame
    is complete."""
    sc = _scene(n, 0.7)
    cam = synth.tiny_camera(200, 150)
    gs = binding.Scene(sc)
    gs.reserve(9_000)
    gs.render(cam)
    torch.cuda.synchronize()
    gk = gs.inspect(binding.RG_INSPECT_KEYS).view(np.uint32).astype(np.uint64)
    gv = gs.inspect(binding.RG_INSPECT_VALUES)
    k, v, _, _ = oracle.keys(sc, cam, oracle.ROOFGS, comp=oracle.compact(sc))
    lay = oracle.layout(cam)
    b_d = np.uint64(lay["b_d"])
    tile = k >> b_d
    tx, ty = tile % np.uint64(lay["tiles_x"]), tile // np.uint64(lay["tiles_x"])
    assert gk.size == 9_000 < k.size
    kept = np.lexsort((tx, v, k & ((np.uint64(1) << b_d) - np.uint64(1)), ty))[:9_000]
    expect = kept[np.lexsort((v[kept], k[kept]))]
    assert np.array_equal(gk, k[expect]) and np.array_equal(gv, v[expect])
    with pytest.raises(binding.RgError) as e:
        gs.check()
    assert e.value.status == 4
    img, st = gs.render(cam, stats=True)
    assert st["regrown"] == 1 and st["n_entries"] == k.size
    full = binding.Scene(sc)
    assert torch.equal(img, full.render(cam, stats=True)[0])


# scales from specks to Gaussians wider than the image, seen from inside the cloud; thin ones; opacities
# around 1/255; every tile shape, and small and larger frames
EXACT_CASES = [(3_000, 0.05, False, (131, 77), (16, 16)), (40_000, 1.0, True, (640, 360), (16, 16)),
               (2_000, 30.0, False, (333, 250), (32, 8)), (2_000, 30.0, True, (250, 333), (8, 32)),
               (500, 300.0, True, (500, 400), (16, 16)), (40_000, 6.0, True, (320, 200), (32, 8)),
               (2_000, 20.0, True, (8192, 48), (16, 16))]


@pytest.mark.parametrize("n,scale,thin,wh,tile", EXACT_CASES)
def test_exact_runs_leave_out_only_pairs_below_the_threshold(n, scale, thin, wh, tile):
    """The timed exact frame leaves out the tiles that a Gaussian reaches below 1/255 everywhere: its
    image equals bit by bit the counting frame's, which keeps every tile of the rectangles, and both
    report the oracle's entries."""
    sc = _scene(n, scale, seed=9)
    rng = np.random.default_rng(1)
    if thin:
        sc.scales[:, 0] *= np.float32(0.01)
    edge = rng.random(n) < 0.4
    sc.opacities[edge] = rng.uniform(0.0, 0.012, int(edge.sum())).astype(np.float32)
    sc.opacities[:2] = (0.0, 1.0)
    cam = synth.look_at_camera((0.1, -0.2, -0.6), *wh, znear=0.02, zfar=5.0, bg=(0.3, 0.2, 0.1))
    gs = binding.Scene(sc, storage=binding.RG_STORE_FP32)
    full, st = gs.render(cam, mode="exact", stats=True, tile=tile)
    k, v, _, _ = oracle.keys(sc, cam, oracle.EXACT, tile=tile)
    ranges = gs.inspect(binding.RG_INSPECT_RANGES)
    assert st["n_entries"] == k.size and 0 < st["n_blends"] < st["n_pairs"]
    for frame in range(2):  # the counting frame, then the timed one
        assert np.array_equal(gs.inspect(binding.RG_INSPECT_KEYS).view(np.uint64), k)
        assert np.array_equal(gs.inspect(binding.RG_INSPECT_VALUES), v)
        assert np.array_equal(gs.inspect(binding.RG_INSPECT_RANGES), ranges)
        img = gs.render(cam, mode="exact", tile=tile)
    assert torch.equal(img, full)
    gs.check()


@pytest.mark.parametrize("n", [1, 31, 1_024, 1_025, 24_577, 311_296, 311_297])
def test_depth_orders(n):
    """Around the sizes where the depth keys' grid changes (one block, 304 blocks of 1,024): many equal
    depth codes (ties by index), culled Gaussians; RoofGS entries equal those of the full 32-bit key
    sort, which orders no Gaussians beforehand, exact ones the oracle's."""
    sc = _scene(n, 1.5 if n < 100_000 else 0.2, seed=n)
    sc.means[: n // 3, 2] = np.float32(0.25)  # equal depths at the camera below
    sc.means[n // 2:: 7, 2] = np.float32(-9.0)  # behind it
    if n > 10:
        sc.opacities[5:: 11] = np.float32(1e-3)
    cam = synth.look_at_camera((0.0, 0.0, -3.0), 200, 120, zfar=4.5)
    gs = binding.Scene(sc)
    gs.render(cam, stats=True)
    a = _entries(gs)
    gs.render(cam, stats=True, flags=binding.RG_FLAG_SORT_FULL_KEY)
    for x, y in zip(a, _entries(gs)):
        assert np.array_equal(x, y)
    gs.render(cam, mode="exact", stats=True)
    k, v, _, _ = oracle.keys(sc, cam, oracle.EXACT)
    assert np.array_equal(gs.inspect(binding.RG_INSPECT_KEYS).view(np.uint64), k)
    assert np.array_equal(gs.inspect(binding.RG_INSPECT_VALUES), v)


# 12,288 tiles and 500,000 Gaussians, the largest frames whose entries are all written, and above them limited ones (the
# first 512 entries of every tile; the last one is too faint for it). Specks: tiles with more than 1,024 entries whose
# pixels are not all finished after 512
LIMIT_CASES = [(500_001, (2048, 1536), (16, 16), 0.4), (500_000, (2048, 1537), (16, 16), 0.4),
               (500_001, (2048, 1537), (16, 16), 0.4), (500_001, (1999, 1777), (32, 8), 0.4),
               (500_001, (1777, 1999), (8, 32), 0.4), (500_001, (2048, 1537), (16, 16), 0.01)]


@pytest.mark.parametrize("n,wh,tile,opacity", LIMIT_CASES)
def test_limited_frames_render_every_entry(n, wh, tile, opacity):
    """Tiles read past the entries written for them are resumed by a second launch: the images equal, bit by bit,
    those of the ordered front end and of the counting launch, and so do the entries that an inspection sees."""
    sc = _scene(n, 0.15, seed=5)
    rng = np.random.default_rng(2)
    sc.opacities = (opacity * rng.uniform(0.9, 1.1, n)).astype(np.float32)
    sc.means[n // 4:] *= np.float32(0.25)  # most of them in the middle
    cam = synth.tiny_camera(*wh, bg=(0.2, 0.1, 0.3))
    gs = binding.Scene(sc)
    for mode in ("roofgs", "exact"):
        gs.render(cam, mode=mode, tile=tile, stats=True)  # sizes the workspace
    for flags in (0, binding.RG_FLAG_QUAD_PIXEL, binding.RG_FLAG_SINGLE_PIXEL | binding.RG_FLAG_EXACT_EXP,
                  binding.RG_FLAG_QUAD_PIXEL | binding.RG_FLAG_EXACT_EXP):
        a = gs.render(cam, flags=flags, tile=tile)
        ea = _entries(gs)
        assert torch.equal(a, gs.render(cam, flags=flags, tile=tile))  # nothing of the inspection is left
        b = gs.render(cam, flags=flags | binding.RG_FLAG_ORDERED_FRONT_END, tile=tile)
        eb = _entries(gs)
        for x, y in zip(ea, eb):
            assert np.array_equal(x, y)
        assert torch.equal(a, b)
    out = torch.empty_like(a)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        gs.render(cam, flags=flags, tile=tile, out=out)
    for _ in range(2):
        out.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(a, out)
    r = ea[2].view(np.uint32).reshape(-1, 2).astype(np.int64)
    assert (r[:, 1] - r[:, 0]).max() > 1_024
    a = gs.render(cam, mode="exact", tile=tile)
    b, _ = gs.render(cam, mode="exact", tile=tile, stats=True)
    b = b.clone()
    assert torch.equal(a, gs.render(cam, mode="exact", tile=tile))
    assert torch.equal(a, b)
    gs.check()


def _specks(cam, tile, n, seed=0):
    """Gaussians about a pixel wide: three of four in the bottom-right tile, the others anywhere in the image."""
    rng = np.random.default_rng(seed)
    lo = np.array([cam.width - tile[0] + 2, cam.height - tile[1] + 2])
    px = rng.uniform(lo, [cam.width - 1, cam.height - 1], size=(n, 2))
    px[::4] = rng.uniform(0, [cam.width - 1, cam.height - 1], size=px[::4].shape)
    z = rng.uniform(2.0, 4.0, n)
    sc = synth.tiny_scene(n, seed=seed)
    sc.means = np.stack([(px[:, 0] - cam.cx) / cam.fx * z, (px[:, 1] - cam.cy) / cam.fy * z, z], 1).astype(np.float32)
    sc.scales = (rng.uniform(0.2, 0.6, (n, 3)) * (z / cam.fx)[:, None]).astype(np.float32)
    return sc


@pytest.mark.parametrize("wh,tile", [((8192, 8192), (16, 16)), ((16384, 4096), (32, 8)), ((4096, 16384), (8, 32))])
def test_the_largest_grid_keeps_its_last_tile(wh, tile):
    """512 x 512 tiles: runs of every lane in the last column of the last row. RoofGS against the ordered front end;
    exact against a view one tile column wider, whose entries are sorted by 64-bit keys (the same Gaussians in the same
    order, so the same pixels)."""
    f = float(wh[0] // 2)
    eye = np.eye(3, dtype=np.float32).reshape(9)

    def camera(w):
        return synth.Camera(eye, np.zeros(3, np.float32), f, f, (wh[0] - 1) / 2.0, (wh[1] - 1) / 2.0, w, wh[1], 0.5, 8.0,
                            np.array([0.2, 0.1, 0.3], np.float32))

    cam = camera(wh[0])
    gs = binding.Scene(_specks(cam, tile, 3_000))
    a, sa = gs.render(cam, stats=True, tile=tile)
    ea = _entries(gs)
    b, sb = gs.render(cam, flags=binding.RG_FLAG_ORDERED_FRONT_END, stats=True, tile=tile)
    eb = _entries(gs)
    last = ea[2].view(np.uint32).reshape(-1, 2)[-1]
    assert int(last[1]) - int(last[0]) > 1_000
    assert torch.equal(a, b)
    for k in ("n_entries", "n_visible", "n_front", "n_pairs", "n_blends"):
        assert sa[k] == sb[k], k
    for x, y in zip(ea, eb):
        assert np.array_equal(x, y)
    a = gs.render(cam, mode="exact", tile=tile)
    b = gs.render(camera(wh[0] + tile[0]), mode="exact", tile=tile)
    assert torch.equal(a, b[:, :, :wh[0]])
    gs.check()


def _ms(gs, cam, out):
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    best = float("inf")
    for _ in range(5):
        a.record()
        for _ in range(10):
            gs.render(cam, out=out)
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


@pytest.mark.parametrize("part", [0.07, 0.5, 0.9])
def test_a_large_frame_beyond_the_capacity(part):
    """Rows of many chunks: the kept entries are the first ones in (tile row, depth code, index, tile column) order of the
    complete frame's, and the frame takes no longer than the complete one (0.5 to 0.95 of it; the bound leaves room for
    noise on a busy machine)."""
    sc = synth.clustered_scene(400_000, 1)
    cam = synth.orbit_camera(0, 1920, 1080, radius=2.5)
    full, small = binding.Scene(sc), binding.Scene(sc)
    _, st = full.render(cam, stats=True)
    k, v, _ = _entries(full)
    k = k.view(np.uint32).astype(np.uint64)
    room = int(k.size * part)
    small.reserve(room)
    out = small.render(cam)
    gk, gv, _ = _entries(small)
    b_d = np.uint64(st["b_d"])
    tx, ty = (k >> b_d) % np.uint64(st["tiles_x"]), (k >> b_d) // np.uint64(st["tiles_x"])
    kept = np.lexsort((tx, v, k & ((np.uint64(1) << b_d) - np.uint64(1)), ty))[:room]
    expect = kept[np.lexsort((v[kept], k[kept]))]
    assert np.array_equal(gk.view(np.uint32), k[expect].astype(np.uint32)) and np.array_equal(gv, v[expect])
    assert _ms(small, cam, out) <= 1.15 * _ms(full, cam, out)


# a small frame, a larger one, a limited one
@pytest.mark.parametrize("n,wh,scale", [(3_000, (200, 150), 2.0), (40_000, (320, 200), 1.0), (520_000, (2064, 1552), 0.5)])
def test_exact_frames_beyond_the_capacity(n, wh, scale):
    """The entries that an exact frame keeps, and blends, are the first ones Gaussian by Gaussian in index order, row by row
    of its rectangle: the image equals that of the scene cut off there, with the last Gaussian in its first tiles only."""
    sc = _scene(n, scale, seed=6)
    cam = synth.tiny_camera(*wh, bg=(0.2, 0.1, 0.3))
    bins = oracle.keys(sc, cam, oracle.EXACT)[3]
    rows, cols = bins[:, 4] - bins[:, 2] + 1, bins[:, 3] - bins[:, 1] + 1
    k = int(np.flatnonzero((np.arange(n) > n // 2) & (bins[:, 0] > 0) & (rows > 1) & (cols > 1))[0])
    sc.opacities[k] = 0.9
    fits = int(cols[k]) + 1  # its first row, and a tile of the second
    room = int(bins[:k, 6].sum()) + fits
    assert room < int(bins[:, 6].sum())
    small = binding.Scene(sc, storage=binding.RG_STORE_FP32)
    small.reserve(room)
    img = small.render(cam, mode="exact")
    want = []
    for m in (k, k + 1):
        gs = binding.Scene(sc.subset(np.arange(m)), storage=binding.RG_STORE_FP32)
        gs.render(cam, mode="exact", stats=True)
        want.append(gs.render(cam, mode="exact").clone())
        gs.close()
    ref = want[0]
    for t in range(fits):
        x, y = 16 * (int(bins[k, 1]) + t % int(cols[k])), 16 * (int(bins[k, 2]) + t // int(cols[k]))
        ref[:, y:y + 16, x:x + 16] = want[1][:, y:y + 16, x:x + 16]
    assert torch.equal(img, ref)
    assert small.inspect(binding.RG_INSPECT_VALUES).size == room
    with pytest.raises(binding.RgError) as e:
        small.check()
    assert e.value.status == 4


@pytest.mark.parametrize("stats", [True, False])
@pytest.mark.parametrize("n", [20_000, 40_000])
def test_inspection_reads_the_device_lists(n, stats):
    """What rg_inspect reports of an exact frame is the counting frame's lists, and for the others is held against the lists
    that the device blends: once a replayed graph has put another frame's in their place, it reports those or refuses."""
    sc = _scene(n)
    cam = synth.tiny_camera(320, 200)
    gs = binding.Scene(sc)
    out = gs.render(cam)
    gs.render(cam, mode="exact", stats=True)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        gs.render(cam, out=out)
    gs.render(cam, mode="exact", stats=stats)
    k, v, r, _ = oracle.keys(sc, cam, oracle.EXACT)
    gk, gv, gr = _entries(gs)
    assert np.array_equal(gk.view(np.uint64), k) and np.array_equal(gv, v)
    assert np.array_equal(gr.view(np.uint32).reshape(-1, 2), r)
    g.replay()
    if stats:
        assert not np.array_equal(gs.inspect(binding.RG_INSPECT_VALUES), v)
    else:
        with pytest.raises(binding.RgError):
            gs.inspect(binding.RG_INSPECT_VALUES)
    gs.render(cam, mode="exact", stats=stats)
    assert np.array_equal(_entries(gs)[1], v)


@pytest.mark.parametrize("mode", ["roofgs", "exact"])
def test_a_replayed_limited_frame_is_inspected_again(mode):
    """A replay leaves values out again, and the state of unfinished tiles in their place: every inspection completes them."""
    n, cam = 500_001, synth.tiny_camera(2048, 1537)
    sc = _scene(n, 0.15, seed=5)
    sc.opacities = np.full(n, 0.4, np.float32)
    sc.means[n // 4:] *= np.float32(0.25)
    gs = binding.Scene(sc)
    out, _ = gs.render(cam, mode=mode, stats=True)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        gs.render(cam, mode=mode, out=out)
    frames = []
    for _ in range(3):
        g.replay()
        frames.append(_entries(gs))
    for f in frames[1:]:
        for x, y in zip(frames[0], f):
            assert np.array_equal(x, y)


def _frame_us(gs, cam, out):
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    best = float("inf")
    for _ in range(4):
        a.record()
        for _ in range(10):
            gs.render(cam, out=out, flags=binding.RG_FLAG_QUAD_PIXEL)
        b.record()
        b.synchronize()
        best = min(best, 100.0 * a.elapsed_time(b))
    return best


def test_limited_frames_of_specks_are_not_slower():
    """Specks of opacity 0.5, two pixels wide, in the middle of a 4K frame: most of their tiles need more than the first 512
    entries, and a frame just above the largest whose entries are all written (500,000 Gaussians) may not pay for a second
    pass over nearly all of them: that cost a quarter; 15 % are allowed for noise and the two launches."""
    rng = np.random.default_rng(0)
    w, h, n = 3840, 2160, 500_002
    cam = synth.Camera(np.eye(3, dtype=np.float32).reshape(9), np.zeros(3, np.float32), w / 2.0, w / 2.0, (w - 1) / 2.0,
                       (h - 1) / 2.0, w, h, 0.5, 50.0)
    sc = synth.tiny_scene(n, seed=0)
    z = rng.uniform(2, 20, n)
    px = np.array([w, h]) / 2 + rng.normal(size=(n, 2)) * 0.02 * np.array([w, h])
    sc.means = np.append((px - [cam.cx, cam.cy]) / cam.fx * z[:, None], z[:, None], 1).astype(np.float32)
    sc.scales = (rng.uniform(1.5, 2.5, (n, 3)) * (z / cam.fx)[:, None]).astype(np.float32)
    sc.opacities = np.full(n, 0.5, np.float32)
    limited, full = binding.Scene(sc), binding.Scene(sc.subset(np.arange(500_000)))
    out, _ = limited.render(cam, stats=True)
    full.render(cam, stats=True)
    assert _frame_us(limited, cam, out) <= 1.15 * _frame_us(full, cam, torch.empty_like(out))


@pytest.mark.parametrize("wh,tile", [((2048, 1552), (16, 16)), ((1999, 1777), (32, 8)), ((1777, 1999), (8, 32))])
def test_limited_frames_resume_unfinished_tiles(wh, tile):
    """Rows that are limited, their left part being opaque soon, with tiles on the right whose pixels are still unfinished after
    every one of their entries: image and entries as the ordered front end's and the counting launch's."""
    rng = np.random.default_rng(4)
    w, h, n = wh[0], wh[1], 600_000
    cam = synth.Camera(np.eye(3, dtype=np.float32).reshape(9), np.zeros(3, np.float32), w / 2.0, w / 2.0, (w - 1) / 2.0,
                       (h - 1) / 2.0, w, h, 0.5, 50.0, np.array([0.2, 0.9, 0.4], np.float32))
    left = np.arange(n) % 3 > 0
    x = np.where(left, rng.uniform(0.05, 0.4, n), rng.uniform(0.55, 0.75, n)) * w
    y = rng.uniform(0.45, 0.55, n) * h
    z, size = rng.uniform(2, 20, n), np.where(left, 5.0, 0.4)  # pixels
    sc = synth.tiny_scene(n, seed=2)
    sc.means = np.stack([(x - cam.cx) / cam.fx * z, (y - cam.cy) / cam.fy * z, z], 1).astype(np.float32)
    sc.scales = np.repeat((size * z / cam.fx)[:, None], 3, 1).astype(np.float32)
    sc.opacities = np.where(left, 0.9, 0.012).astype(np.float32)
    # the optical depth that 512 entries bring, as the rule estimates it, in the rows between 0.46 and 0.54 of the height: far
    # above its 12
    s2, o = size ** 2 + 0.3, sc.opacities.astype(np.float64)
    box = 2 * np.sqrt(2 * np.log(255 * o) * s2)
    tiles = (box / tile[0] + 1) * (box / tile[1] + 1)
    depth = 2 * np.pi * s2 * sum(o ** k / k ** 2 for k in range(1, 60)) / 256
    for r in np.linspace(0.46, 0.54, 9):
        row = np.abs(y - r * h) < 16
        assert 512 * depth[row].sum() / tiles[row].sum() > 20
    gs = binding.Scene(sc)
    for flags in (0, binding.RG_FLAG_QUAD_PIXEL, binding.RG_FLAG_SINGLE_PIXEL | binding.RG_FLAG_EXACT_EXP):
        gs.render(cam, flags=flags, tile=tile, stats=True)
        a = gs.render(cam, flags=flags, tile=tile)
        ea = _entries(gs)
        b = gs.render(cam, flags=flags | binding.RG_FLAG_ORDERED_FRONT_END, tile=tile)
        for p, q in zip(ea, _entries(gs)):
            assert np.array_equal(p, q)
        assert torch.equal(a, b)
    b, st = gs.render(cam, mode="exact", tile=tile, stats=True)
    r = gs.inspect(binding.RG_INSPECT_RANGES).reshape(-1, 2).astype(np.int64)
    per_tile = (r[:, 1] - r[:, 0]).reshape(st["tiles_y"], st["tiles_x"])
    a = gs.render(cam, mode="exact", tile=tile).clone()
    assert torch.equal(a, b)
    # unfinished: the background shows through
    cam.bg = np.zeros(3, np.float32)
    through = (a - gs.render(cam, mode="exact", tile=tile))[1].cpu().numpy() / 0.9
    ty, tx = int(0.5 * h) // tile[1], int(0.65 * w) // tile[0]
    assert per_tile[ty, tx] > 512
    assert through[ty * tile[1]:(ty + 1) * tile[1], tx * tile[0]:(tx + 1) * tile[0]].max() > 1e-2
    gs.check()


@pytest.mark.parametrize("cols", [127, 128, 129, 136, 137, 256, 257])
def test_windows_of_columns(cols):
    """Grids about a window of the expansion (128 tile columns) and two, a small frame and a larger one: entries and image as the
    ordered front end's."""
    cam = synth.tiny_camera(16 * cols - 3, 90, bg=(0.2, 0.1, 0.3))
    for n in (6_000, 36_000):
        gs = binding.Scene(_scene(n, 2.0, seed=cols))
        gs.render(cam, stats=True)
        a = gs.render(cam)
        ea = _entries(gs)
        assert torch.equal(a, gs.render(cam, flags=binding.RG_FLAG_ORDERED_FRONT_END))
        for x, y in zip(ea, _entries(gs)):
            assert np.array_equal(x, y)
