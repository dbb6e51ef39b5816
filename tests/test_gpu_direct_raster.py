"""The routes a frame takes by its triangles' sizes, against the oracle: small
triangles rasterized by the count pass into one key per pixel, medium boxes
shared out by rows and samples, large ones by a warp each.  Keys bit for bit,
colours within 1e-5 (the tolerance of the other parity tests), and the bin
lists' size as with every triangle binned."""
import numpy as np
import pytest

import oracle
from paper_1404_6293_gb300 import scenes as S

pytestmark = pytest.mark.gpu

RGB_TOL = 1e-5


def _torch():
    import torch
    return torch


def _frame(r, s):
    torch = _torch()
    from paper_1404_6293_gb300.raster import DeviceScene
    fb = r.forward(DeviceScene.from_host(s))
    torch.cuda.synchronize()
    code, need = r.status()
    assert code == 0
    return fb, need


def _check(s, bins=16, schedule="static"):
    """Oracle parity of the default route, and of every triangle binned."""
    from paper_1404_6293_gb300 import _lib as L
    from paper_1404_6293_gb300.raster import Rasterizer
    ref, st = oracle.raster_bbox(s, threads=8)
    assert st == 0
    r = Rasterizer(s.width, s.height, bins, bins, schedule)
    rb = Rasterizer(s.width, s.height, bins, bins, schedule)
    rb.set_option(L.PIKO_OPT_SMALL_TRI_PIXELS, 0)  # no direct rasterization
    fb, need = _frame(r, s)
    fbb, need_binned = _frame(rb, s)
    assert need == need_binned
    for f in (fb, fbb):
        assert np.array_equal(f.key_numpy(), ref)
        if s.shade_mode != S.SHADE_GBUFFER:
            assert np.abs(f.rgba.cpu().numpy() - oracle.shade(s, ref)).max() <= RGB_TOL
    return r


def _triangles(W, H, boxes, seed, copies=1):
    """Right triangles in both windings whose snapped bounding boxes start at
    16.8 positions x, y and measure w, h pixels (fractions of 1/256 allowed)."""
    rng = np.random.default_rng(seed)
    pos = []
    for k in range(copies):
        for (w, h) in boxes:
            x0 = np.rint(rng.uniform(-2, max(W - w, 1)) * 256) / 256
            y0 = np.rint(rng.uniform(-2, max(H - h, 1)) * 256) / 256
            c = [(x0, y0), (x0 + w, y0), (x0, y0 + h)]
            if rng.random() < 0.5:
                c = [(x0 + w, y0 + h), (x0, y0 + h), (x0 + w, y0)]
            if rng.random() < 0.5:
                c = c[::-1]
            for (x, y) in c:
                pos.append((x / W * 2 - 1, 1 - y / H * 2, rng.uniform(-0.9, 0.9), 1.0))
    n = len(pos)
    return S.Scene(W, H, np.asarray(pos, np.float32), np.arange(n, dtype=np.int32).reshape(-1, 3),
                   color=rng.uniform(0, 1, (n, 3)).astype(np.float32))


# boxes around the limits: 32 samples in every shape, one more, a column or row
# of 32 and 33, and extents around 128 pixels
_LIMITS = [(32, 1), (33, 1), (1, 32), (1, 33), (8, 4), (4, 8), (16, 2), (11, 3), (2, 17), (0.5, 0.5), (1 / 256, 40),
           (127 + 255 / 256, 0.4), (128, 0.4), (0.4, 127 + 255 / 256), (0.4, 128), (6, 6), (30, 30), (63, 20),
           (127.5, 90), (90, 129)]


@pytest.mark.parametrize("bins", [8, 16, 32, 64])
@pytest.mark.parametrize("size", [(131, 137), (150, 70)])
def test_boxes_at_the_limits(bins, size):
    W, H = size
    copies = -(-W * H // (4 * len(_LIMITS))) + 1  # enough triangles for the direct route
    _check(_triangles(W, H, _LIMITS, 7 * bins + W, copies), bins, "dynamic").close()


@pytest.mark.parametrize("mode,color", [(S.SHADE_LAMBERT, True), (S.SHADE_LAMBERT, False), (S.SHADE_GOURAUD, True),
                                        (S.SHADE_GBUFFER, True)])
@pytest.mark.parametrize("size", [(1, 1), (8, 3), (257, 63), (640, 361)])
def test_tiny_triangles_in_every_mode(mode, color, size):
    W, H = size
    q = max(2, int(np.sqrt(W * H / 3.0)))
    s = S.heightfield(W, H, q, q, seed=W + H, with_color=True)
    if mode != S.SHADE_LAMBERT:
        s.shade_mode = mode
    if not color:
        s.color = None
    _check(s, 8 if W < 16 else 16, "hardware").close()


def test_mixed_sizes_without_the_capacity_check_and_across_frames():
    """One handle: frames whose bin lists grow at the same triangle count (the
    second overflows the first's lists behind the launched stages), and the
    check turned off afterwards."""
    from paper_1404_6293_gb300 import _lib as L
    from paper_1404_6293_gb300.raster import Rasterizer
    W, H, T = 200, 150, 3000
    scenes = [S.random_triangles(W, H, T, radius, seed=11 + k) for k, radius in enumerate((2.0, 3.0, 60.0, 2.0, 25.0))]
    r = Rasterizer(W, H, 8, 8, "static")
    for check in (1, 0):
        r.set_option(L.PIKO_OPT_CHECK_CAPACITY, check)
        for s in scenes:
            ref, _ = oracle.raster_bbox(s, threads=8)
            fb, _ = _frame(r, s)
            assert np.array_equal(fb.key_numpy(), ref)
            assert np.abs(fb.rgba.cpu().numpy() - oracle.shade(s, ref)).max() <= RGB_TOL
    r.close()


def test_overflow_of_a_direct_frame_writes_nothing():
    """A frame of directly rasterized triangles overflows at the size its bin
    lists would have had, and leaves no trace in the next frame."""
    torch = _torch()
    from paper_1404_6293_gb300 import _lib as L
    from paper_1404_6293_gb300.raster import DeviceScene, Framebuffer, Rasterizer
    s = S.heightfield(128, 96, 80, 60, seed=3)
    small = S.heightfield(128, 96, 40, 20, seed=4)
    r = Rasterizer(128, 96, 8, 8, "dynamic")
    r.reserve(s.num_vertices, s.num_triangles, 3000)  # room for 4,774 entries (a quarter and 1,024 more)
    r.set_option(L.PIKO_OPT_CHECK_CAPACITY, 0)
    _frame(r, small)
    fb = Framebuffer.allocate(128, 96, s.shade_mode)
    fb.key.fill_(7)
    fb.rgba.fill_(-1.0)
    r.forward(DeviceScene.from_host(s), fb)
    torch.cuda.synchronize()
    code, need = r.status()
    assert code == L.PIKO_ERR_OVERFLOW and need > 4774
    assert bool((fb.key == 7).all()) and bool((fb.rgba == -1.0).all())
    fb2, _ = _frame(r, small)
    assert np.array_equal(fb2.key_numpy(), oracle.raster_bbox(small)[0])
    r.close()


@pytest.mark.parametrize("check", [0, 1])
def test_batch_of_all_routes(check):
    torch = _torch()
    from paper_1404_6293_gb300 import _lib as L
    from paper_1404_6293_gb300.raster import DeviceScene, Rasterizer
    scenes = [S.heightfield(100, 75, 60, 50, seed=1, with_color=True), S.random_triangles(90, 60, 40, 30.0, seed=2),
              S.random_triangles(33, 200, 2000, 4.0, seed=3), _triangles(131, 137, _LIMITS, 4, 230),
              S.power_law_triangles(120, 90, 2000, seed=5)]
    r = Rasterizer(100, 75, 16, 16, "static")
    ds = [DeviceScene.from_host(s) for s in scenes]
    r.forward_batch(ds)
    r.set_option(L.PIKO_OPT_CHECK_CAPACITY, check)
    fbs = r.forward_batch(ds, None, [(16, 16), (8, 8), (32, 16), (64, 64), (16, 32)],
                          ["static", "dynamic", "static", "dynamic", "hardware"])
    torch.cuda.synchronize()
    assert r.status()[0] == 0
    for s, fb in zip(scenes, fbs):
        ref, _ = oracle.raster_bbox(s, threads=8)
        assert np.array_equal(fb.key_numpy(), ref)
        if s.shade_mode != S.SHADE_GBUFFER:
            assert np.abs(fb.rgba.cpu().numpy() - oracle.shade(s, ref)).max() <= RGB_TOL
    r.close()


# Sums of n float32 terms in any order differ by at most n 2^-24 sum |term|
# (first order), and each term by a few roundings; 1e-4 of the largest gradient
# is the gradient contract of the other tests.
def _close(a, b):
    a, b = a.cpu().numpy().astype(np.float64), b.cpu().numpy().astype(np.float64)
    assert np.abs(a - b).max() <= 1e-4 * max(np.abs(b).max(), 1e-30)


@pytest.mark.parametrize("quads", [(60, 40), (6, 5)])  # tiny and large triangles
@pytest.mark.parametrize("color", [True, False])
def test_stored_gradients_equal_added_ones(quads, color):
    torch = _torch()
    from paper_1404_6293_gb300.raster import DeviceScene, Rasterizer
    s = S.heightfield(97, 61, *quads, seed=8, with_color=True)
    ds = DeviceScene.from_host(s)
    if not color:
        ds.color = None
    r = Rasterizer(97, 61)
    fb = r.forward(ds)
    g = torch.randn((61, 97, 4), device="cuda", generator=torch.Generator("cuda").manual_seed(5))
    dc, dn, dl = (torch.zeros((s.num_vertices, 3), device="cuda"), torch.zeros_like(ds.normal),
                  torch.zeros_like(ds.light_dir))
    r.backward(ds, fb, g, dc, dn, dl)
    r.backward(ds, fb, g, dc, dn, dl)  # added: twice the gradient
    junk = [torch.full_like(t, float("nan")) for t in (dc, dn, dl)]  # freed, so that new tensors hold them
    del junk
    gc, gn, gl = r.gradients(ds, fb, g, color=color)
    torch.cuda.synchronize()
    if color:
        _close(2 * gc, dc)
    else:
        assert gc is None and not dc.any()
    _close(2 * gn, dn)
    _close(2 * gl, dl)
    ds.tris = ds.tris[:0].contiguous()
    for t in r.gradients(ds, fb, g, color=color):
        assert t is None or not t.any()
    r.close()


def test_batch_gradients_with_shared_and_own_arrays():
    """Scenes that share gradient arrays, in a row and apart, add into them."""
    torch = _torch()
    from paper_1404_6293_gb300.raster import DeviceScene, Rasterizer
    base, mvps = S.sphere_views(4, 96, 80, 24, 18, seed=2)
    other = S.heightfield(70, 90, 40, 30, seed=6, with_color=True)
    import dataclasses
    views = [DeviceScene.from_host(dataclasses.replace(base, mvp=m)) for m in mvps]
    for v in views[1:]:
        v.pos, v.tris, v.color, v.normal, v.light_dir = (views[0].pos, views[0].tris, views[0].color, views[0].normal,
                                                        views[0].light_dir)
    scenes = [views[0], views[1], DeviceScene.from_host(other), views[2], views[3]]
    r = Rasterizer(96, 80)
    fbs = r.forward_batch(scenes)
    gen = torch.Generator("cuda").manual_seed(9)
    gs = [torch.randn((s.height, s.width, 4), device="cuda", generator=gen) for s in scenes]

    def arrays():
        m = [torch.zeros_like(t) for t in (views[0].color, views[0].normal, views[0].light_dir)]
        o = [torch.zeros_like(t) for t in (scenes[2].color, scenes[2].normal, scenes[2].light_dir)]
        return m, o, [[(o if k == 2 else m)[j] for k in range(5)] for j in range(3)]

    m, o, lists = arrays()
    r.backward_batch(scenes, fbs, gs, *lists)
    sm, so, slists = arrays()
    for k, s in enumerate(scenes):
        rs = Rasterizer(s.width, s.height)
        rs.backward(s, fbs[k], gs[k], *[slists[j][k] for j in range(3)])
        torch.cuda.synchronize()
        rs.close()
    for a, b in zip(m + o, sm + so):
        _close(a, b)
    r.close()


@pytest.mark.parametrize("n", [1, 2, 5])
@pytest.mark.parametrize("far", [False, True])
def test_light_pairs_and_single_lights(n, far):
    """Odd and even counts, with and without a light outside the paired form's
    range (far away, or not finite and behind every pixel)."""
    torch = _torch()
    from paper_1404_6293_gb300.raster import Framebuffer, Rasterizer
    W, H = 61, 45
    key, gn, ga = S.gbuffer_inputs(W, H)
    lights = S.point_lights(W, H, n)
    if far:
        lights[n - 1, :3] = (1e7, -2e7, -1e7)
    ref = oracle.light_pass(key, gn.view(np.uint16), ga.view(np.uint16), lights)
    r = Rasterizer(W, H)
    fb = Framebuffer(torch.from_numpy(key.view(np.int64)).cuda(), None, torch.from_numpy(gn).cuda(),
                     torch.from_numpy(ga).cuda())
    out = r.deferred_light(fb, torch.from_numpy(lights).cuda()).cpu().numpy()
    assert np.abs(out - ref).max() <= RGB_TOL
    r.close()
