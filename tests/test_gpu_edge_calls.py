"""Calls at the edges of what the entry points accept: scenes without
triangles or normals, odd light counts, attribute arrays longer than the
scene, scratch reserved ahead of a capture, and replayed graphs whose inputs
change between replays."""
import ctypes as C
import dataclasses

import numpy as np
import pytest

import oracle
from paper_1404_6293_gb300 import scenes as S

pytestmark = pytest.mark.gpu

EMPTY = -1  # the all-ones key, as int64


def _torch():
    import torch
    return torch


def _bare_lambert(W, H, color):
    """A Lambert scene of 300 vertices, no triangles and no normals."""
    from paper_1404_6293_gb300.raster import DeviceScene
    s = S.heightfield(W, H, 24, 11, seed=2, with_color=True)
    ds = DeviceScene.from_host(s)
    assert ds.num_vertices == 300 and ds.shade_mode == S.SHADE_LAMBERT
    ds.tris = ds.tris[:0].contiguous()
    ds.normal = None
    if not color:
        ds.color = None
    return ds


@pytest.mark.parametrize("color", [True, False])
def test_lambert_scene_without_triangles_needs_no_normals(color):
    """Every call that takes a scene: an empty frame, and no gradient."""
    torch = _torch()
    from paper_1404_6293_gb300 import _lib as L
    from paper_1404_6293_gb300.raster import DeviceScene, Framebuffer, HostScene, Rasterizer
    W, H = 64, 48
    ds = _bare_lambert(W, H, color)
    r = Rasterizer(W, H)

    def check(fb, what):
        torch.cuda.synchronize()
        assert r.status()[0] == 0, what
        assert bool((fb.key == EMPTY).all()) and not bool(fb.rgba.any()), what

    for check_capacity in (1, 0):
        r.set_option(L.PIKO_OPT_CHECK_CAPACITY, check_capacity)
        check(r.forward(ds), "forward")
    r.set_option(L.PIKO_OPT_CHECK_CAPACITY, 1)
    full = S.heightfield(W, H, 30, 20, seed=3, with_color=True)
    dfull = DeviceScene.from_host(full)
    fbs = r.forward_batch([dfull, ds])
    check(fbs[1], "batch")
    assert np.array_equal(fbs[0].key_numpy(), oracle.raster_bbox(full)[0])

    hs = HostScene.from_host(full)
    hs.tris, hs.normal = hs.tris[:0].contiguous(), None
    check(r.forward_host(hs), "host")

    fb = Framebuffer.allocate(W, H, ds.shade_mode)
    status = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    f = L.load().piko_raster_forward_noalloc
    f.argtypes = [C.POINTER(L.PikoScene), C.POINTER(L.PikoFramebuffer), C.c_int, C.c_int, C.c_int, C.c_void_p,
                  C.c_void_p]
    f.restype = C.c_int
    cs, cf = ds.c_struct(), fb.c_struct()
    assert f(C.byref(cs), C.byref(cf), 16, 16, 0, C.c_void_p(status.data_ptr()),
             C.c_void_p(torch.cuda.current_stream().cuda_stream)) == L.PIKO_OK
    check(fb, "without allocation")
    assert int(status.item()) == L.PIKO_OK

    g = torch.ones((H, W, 4), device="cuda")
    dc = torch.full((ds.num_vertices, 3), 2.0, device="cuda")
    dl = torch.full((3,), 2.0, device="cuda")
    r.backward(ds, fb, g, dc if color else None, None, dl)
    gc, gn, gl = r.gradients(ds, fb, g, color=color, normal=False)
    r.backward_batch([dfull, ds], fbs, [g, g], [None, dc if color else None], None, [None, dl])
    torch.cuda.synchronize()
    assert bool((dc == 2.0).all()) and bool((dl == 2.0).all())  # added to: nothing
    assert gn is None and not bool(gl.any()) and (gc is None or not bool(gc.any()))
    r.close()


@pytest.mark.parametrize("n", [1, 2, 3, 64, 65])
def test_light_pass_with_an_infinite_normal(n):
    """A binary16 normal that overflowed gives an infinite sum where a light
    shines on it and nothing where none does, for odd and even counts; never
    NaN.  Other pixels are the oracle's."""
    torch = _torch()
    from paper_1404_6293_gb300.raster import Framebuffer, Rasterizer
    W, H = 61, 45
    key, gn, ga = S.gbuffer_inputs(W, H, empty_frac=0.0)
    lights = S.point_lights(W, H, n)
    lights[:, 2] = -5.0  # on the viewer's side of every sample
    facing, away = (7, 11), (30, 20)
    gn[facing] = (0.0, 0.0, -np.inf, 0.0)
    gn[away] = (0.0, 0.0, np.inf, 0.0)
    finite = gn.copy()
    finite[facing] = finite[away] = 0
    ref = oracle.light_pass(key, finite.view(np.uint16), ga.view(np.uint16), lights)
    r = Rasterizer(W, H)
    fb = Framebuffer(torch.from_numpy(key.view(np.int64)).cuda(), None, torch.from_numpy(gn).cuda(),
                     torch.from_numpy(ga).cuda())
    out = r.deferred_light(fb, torch.from_numpy(lights).cuda()).cpu().numpy()
    assert (ga[facing][:3] > 0).all() and (lights[:, 3] > 0).all()
    assert np.isposinf(out[facing][:3]).all()
    assert (out[away][:3] == 0.0).all()
    out[facing] = ref[facing]
    assert np.abs(out - ref).max() <= 1e-5
    r.close()


def test_reserve_covers_the_keys_of_every_mesh_within_the_sizes():
    """Sizes with two vertices a triangle and more, of which a mesh at 4 to 16
    pixels a triangle makes up a part: its forward allocates nothing and is
    captured as it runs uncaptured."""
    torch = _torch()
    from paper_1404_6293_gb300 import _lib as L
    from paper_1404_6293_gb300.raster import DeviceScene, Framebuffer, Rasterizer
    W, H = 1280, 1024  # 10 MB of keys
    s = S.heightfield(W, H, 400, 200, seed=12, with_color=True)
    T = s.num_triangles
    assert 4 * T < W * H <= 16 * T and s.num_vertices < 2 * T
    ds = DeviceScene.from_host(s)
    ref = oracle.raster_bbox(s, threads=8)[0]
    fb = Framebuffer.allocate(W, H, s.shade_mode)
    warm = Rasterizer(W, H)  # loads the kernels
    warm.forward(ds, fb)
    warm.set_option(L.PIKO_OPT_CHECK_CAPACITY, 0)
    warm.forward(ds, fb)
    torch.cuda.synchronize()
    assert warm.status()[0] == 0
    r = Rasterizer(W, H)
    r.reserve(2 * T, T, 4 * T)
    r.set_option(L.PIKO_OPT_CHECK_CAPACITY, 0)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    fb.key.fill_(0)
    r.forward(ds, fb)
    torch.cuda.synchronize()
    assert r.status()[0] == 0
    assert np.array_equal(fb.key_numpy(), ref)
    assert torch.cuda.mem_get_info()[0] == free
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        r.forward(ds, fb)
    fb.key.fill_(0)
    g.replay()
    torch.cuda.synchronize()
    assert np.array_equal(fb.key_numpy(), ref)
    r.close()
    warm.close()


def _cameras(n):
    """Zooms and shifts of the identity camera, each unlike the one before it."""
    out = []
    for k in range(n):
        m = np.eye(4, dtype=np.float32)
        m[0, 0] = m[1, 1] = (1.0, 0.3, 1.6, 0.7, 2.0, 0.5)[k % 6]
        m[0, 3], m[1, 3] = 0.4 * np.cos(2.0 * k), 0.4 * np.sin(2.0 * k)
        out.append(m.ravel())
    return out


@pytest.mark.parametrize("schedule", ["static", "dynamic"])
@pytest.mark.parametrize("kind", ["binned", "direct"])
def test_replays_of_a_captured_frame_follow_the_camera(kind, schedule):
    """16,384 bins (eight scan chunks, which look back at each other) and
    triangles across hundreds of them, captured once and replayed with another
    camera each time: every replay is the oracle's frame."""
    torch = _torch()
    from paper_1404_6293_gb300 import _lib as L
    from paper_1404_6293_gb300.raster import DeviceScene, Framebuffer, Rasterizer
    W = H = 1024
    large = S.random_triangles(W, H, 60, 400.0, seed=31)
    if kind == "binned":
        s = S.random_triangles(W, H, 3000, 12.0, seed=32)
    else:
        s = S.random_triangles(W, H, 400000, 2.0, seed=33)
    pos = np.concatenate([s.pos, large.pos])
    s = S.Scene(W, H, pos, np.arange(len(pos), dtype=np.int32).reshape(-1, 3),
                color=np.concatenate([s.color, large.color]), mvp=np.eye(4, dtype=np.float32).ravel())
    ds = DeviceScene.from_host(s)
    fb = Framebuffer.allocate(W, H, s.shade_mode)
    r = Rasterizer(W, H, 8, 8, schedule)
    r.reserve(s.num_vertices, s.num_triangles, 4_000_000)
    r.set_option(L.PIKO_OPT_CHECK_CAPACITY, 0)
    r.forward(ds, fb)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        r.forward(ds, fb)
    for k, m in enumerate(_cameras(7)):
        ds.mvp.copy_(torch.from_numpy(m))
        fb.key.fill_(0)
        for _ in range(1 + k % 2):  # (also twice without a change)
            g.replay()
        torch.cuda.synchronize()
        assert r.status()[0] == 0
        ref = oracle.raster_bbox(dataclasses.replace(s, mvp=m), threads=8)[0]
        assert np.array_equal(fb.key_numpy(), ref), f"replay {k}"
    ref = oracle.raster_bbox(s, threads=8)[0]  # an ordinary call among the replays
    ds.mvp.copy_(torch.from_numpy(s.mvp))
    r.forward(ds, fb)
    torch.cuda.synchronize()
    assert np.array_equal(fb.key_numpy(), ref)
    r.close()


@pytest.mark.parametrize("launch", [0, 1])
def test_replays_of_a_captured_batch_follow_the_cameras(launch):
    """12,288 bins of three scenes: a dozen scan chunks."""
    torch = _torch()
    from paper_1404_6293_gb300 import _lib as L
    from paper_1404_6293_gb300.raster import DeviceScene, Rasterizer
    W = H = 512
    host = [S.random_triangles(W, H, 2000, 9.0, seed=41), S.random_triangles(W, H, 100000, 2.0, seed=42),
            S.random_triangles(W, H, 100, 150.0, seed=43)]
    host = [dataclasses.replace(s, mvp=np.eye(4, dtype=np.float32).ravel()) for s in host]
    ds = [DeviceScene.from_host(s) for s in host]
    r = Rasterizer(W, H, 8, 8)
    r.set_option(L.PIKO_OPT_BATCH_LAUNCH, launch)
    cams = _cameras(6)
    big = torch.from_numpy(cams[4])  # the most bin entries: sizes the lists
    for d in ds:
        d.mvp.copy_(big)
    fbs = r.forward_batch(ds)
    for m in cams:
        for d in ds:
            d.mvp.copy_(torch.from_numpy(m))
        r.forward_batch(ds, fbs)
    r.set_option(L.PIKO_OPT_CHECK_CAPACITY, 0)
    r.forward_batch(ds, fbs)
    torch.cuda.synchronize()
    assert r.status()[0] == 0
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        r.forward_batch(ds, fbs)
    for k in range(7):
        for i, d in enumerate(ds):
            d.mvp.copy_(torch.from_numpy(cams[(k + i) % 6]))
        for _ in range(1 + k % 2):
            g.replay()
        torch.cuda.synchronize()
        assert r.status()[0] == 0
        for i, s in enumerate(host):
            ref = oracle.raster_bbox(dataclasses.replace(s, mvp=cams[(k + i) % 6]), threads=8)[0]
            assert np.array_equal(fbs[i].key_numpy(), ref), f"replay {k}, scene {i}"
    r.close()


def test_gradients_of_arrays_longer_than_the_scene():
    """Attribute arrays padded past the scene's vertices (a buffer reused for
    several meshes): the padding's gradient is zero through autograd."""
    torch = _torch()
    from paper_1404_6293_gb300.autograd import render
    from paper_1404_6293_gb300.raster import DeviceScene, Rasterizer
    s = S.heightfield(97, 61, 30, 20, seed=8, with_color=True)
    ds = DeviceScene.from_host(s)
    V, r = s.num_vertices, Rasterizer(97, 61)

    def padded(t, rows):
        return torch.cat([t, torch.ones((rows,) + tuple(t.shape[1:]), device="cuda")]).requires_grad_(True)

    g = torch.randn((61, 97, 4), device="cuda", generator=torch.Generator("cuda").manual_seed(5))
    plain = [t.clone().requires_grad_(True) for t in (ds.color, ds.normal, ds.light_dir)]
    long = [padded(ds.color, 400), padded(ds.normal, 400), padded(ds.light_dir, 2)]
    want = torch.autograd.grad(render(r, ds, *plain)[0], plain, g)
    rgba = render(r, ds, *long)[0]
    junk = [torch.full_like(t, float("nan")) for t in long]  # freed, so that new tensors hold them
    del junk
    got = torch.autograd.grad(rgba, long, g)
    torch.cuda.synchronize()
    for a, b, n in zip(got, want, (V, V, 3)):
        assert not bool(a[n:].any())
        assert float((a[:n] - b).abs().max()) <= 1e-4 * float(b.abs().max())
    r.close()


def test_batch_launch_option_selects_the_form():
    """PIKO_OPT_BATCH_LAUNCH: one kernel for 0, one per phase for 1 and by
    default, with the same keys (tests that compare the two rely on it)."""
    torch = _torch()
    from torch.profiler import ProfilerActivity, profile
    from paper_1404_6293_gb300 import _lib as L
    from paper_1404_6293_gb300.raster import DeviceScene, Rasterizer
    ds = [DeviceScene.from_host(s) for s in (S.random_triangles(160, 120, 500, 20.0, seed=51),
                                             S.heightfield(200, 150, 90, 70, seed=52))]
    keys, names = [], []
    with profile(activities=[ProfilerActivity.CUDA]):  # (a process's first session may miss its kernels)
        torch.zeros(8, device="cuda")
        torch.cuda.synchronize()
    for launch in (None, 0, 1):
        r = Rasterizer(64, 64, 8, 8)
        if launch is not None:
            r.set_option(L.PIKO_OPT_BATCH_LAUNCH, launch)
        r.forward_batch(ds)
        with profile(activities=[ProfilerActivity.CUDA]) as p:
            fbs = r.forward_batch(ds)
            torch.cuda.synchronize()
        assert r.status()[0] == 0
        keys.append([f.key.clone() for f in fbs])
        found = " ".join(e.name for e in p.events())
        names.append({k for k in ("k_batch_forward", "k_batch_count", "k_batch_process") if k in found})
        r.close()
    per_phase = {"k_batch_count", "k_batch_process"}
    assert names == [per_phase, {"k_batch_forward"}, per_phase]
    for k in keys[1:]:
        assert all(torch.equal(a, b) for a, b in zip(k, keys[0]))


def _pixel_triangles(W, H, corners, order):
    """A triangle per pixel of a W x H frame (powers of two), its corners at
    offsets (1/256 pixel) from the pixel's centre, in the vertex array at
    order[t] + (0, 1, 2)."""
    y, x = np.divmod(np.arange(W * H), W)
    c = np.stack([x + 0.5, y + 0.5], 1)[:, None, :] + np.asarray(corners, np.float64) / 256.0
    pos = np.zeros((int(order[-1]) + 3, 4), np.float32)
    tris = (order[:, None] + np.arange(3)).astype(np.int32)
    pos[:, 3] = 1.0
    pos[tris, 0] = c[..., 0] * (2.0 / W) - 1.0
    pos[tris, 1] = 1.0 - c[..., 1] * (2.0 / H)
    return pos, tris


def test_gradient_weights_are_correctly_rounded():
    """dL/dc of a vertex of a one-pixel Gouraud triangle under dL/drgb = 1 is the
    pixel's weight: the correctly rounded quotient of its edge function and the
    triangle's area."""
    torch = _torch()
    from paper_1404_6293_gb300.raster import DeviceScene, Rasterizer
    W, H = 64, 32
    T = W * H
    rng = np.random.default_rng(6)
    # around the centre, in three sectors, so that it is inside; all distinct
    ang = np.array([0.3, 2.4, 4.5]) + rng.uniform(-0.4, 0.4, (T, 3))
    rad = rng.uniform(40, 120, (T, 3))
    off = np.rint(np.stack([rad * np.cos(ang), rad * np.sin(ang)], -1)).astype(np.int64)
    pos, tris = _pixel_triangles(W, H, off, np.arange(0, 3 * T, 3))
    s = S.Scene(W, H, pos, tris, color=np.ones((3 * T, 3), np.float32))
    ds, r = DeviceScene.from_host(s), Rasterizer(W, H)
    fb = r.forward(ds)
    torch.cuda.synchronize()
    assert np.array_equal(fb.key_numpy().ravel() & 0xFFFFFFFF, np.arange(T))
    dc, _, _ = r.gradients(ds, fb, torch.ones((H, W, 4), device="cuda"), normal=False, light=False)

    def cross(a, b):
        return a[:, 0] * b[:, 1] - a[:, 1] * b[:, 0]

    w = np.stack([cross(off[:, 1], off[:, 2]), cross(off[:, 2], off[:, 0]), cross(off[:, 0], off[:, 1])], 1)
    A = w.sum(1, keepdims=True)
    want = (w.astype(np.float64) / A).astype(np.float32)  # (both below 2^17: no double rounding)
    got = dc.cpu().numpy().reshape(T, 3, 3)
    for c in range(3):
        assert np.array_equal(got[:, :, c], want)
    r.close()


def test_light_gradient_of_a_fine_mesh_adds_few_terms():
    """524,288 vertices of which every 256 hold one visible triangle with the same
    light gradient r: 2,048 r to within one rounding (at most 2^-24 of a sum
    that grows to the total, half of it on average) for each of 256 additions.
    An addition per 256 vertices is off by 1.1e-5 to 2.1e-5 for most r."""
    torch = _torch()
    from paper_1404_6293_gb300.raster import DeviceScene, Rasterizer
    W, H = 64, 32
    T = W * H
    # weights 1/4, 1/4 and 1/2 at the centre, and every product below exact
    pos, tris = _pixel_triangles(W, H, [(-64, 32), (64, 32), (0, -32)], 256 * np.arange(T))
    V = 256 * T
    pos = np.concatenate([pos, np.tile(np.float32([0, 0, 0, 1]), (V - len(pos), 1))])
    r = Rasterizer(W, H)
    for a, b in ((1.3, 1.7), (0.9, 1.05), (1.9, 0.7)):
        n = np.tile(np.float32([a, b, 1.0]), (V, 1))
        s = S.Scene(W, H, pos, tris, color=np.ones((V, 3), np.float32), normal=n,
                    light_dir=np.float32([0.0, 0.0, 1.0]), shade_mode=S.SHADE_LAMBERT)
        ds = DeviceScene.from_host(s)
        fb = r.forward(ds)
        g = torch.zeros((H, W, 4), device="cuda")
        g[..., 0] = 1.0
        _, _, dl = r.gradients(ds, fb, g, color=False, normal=False)
        assert int((fb.key != EMPTY).sum()) == T
        want = T * n[0].astype(np.float64)
        assert (np.abs(dl.cpu().numpy() - want) <= 256 * 2.0 ** -25 * want).all()
    r.close()


def test_batch_light_gradient_of_groups_that_share_ctas():
    """Scenes of very uneven size with arrays of their own: the finishing pass deals
    their vertices out in chunks, several groups to a CTA and several CTAs to a
    group.  Each light gradient is 64 or 2,048 equal terms."""
    torch = _torch()
    from paper_1404_6293_gb300.raster import DeviceScene, Rasterizer
    host = []
    for k, (W, H, step) in enumerate([(64, 32, 256), (8, 8, 3), (8, 8, 40), (64, 32, 3), (8, 8, 3), (64, 32, 700),
                                      (8, 8, 5)]):
        T = W * H
        pos, tris = _pixel_triangles(W, H, [(-64, 32), (64, 32), (0, -32)], step * np.arange(T))
        n = np.tile(np.float32([0.25 * (k + 1), 1.5, 1.0]), (len(pos), 1))
        host.append(S.Scene(W, H, pos, tris, color=np.ones((len(pos), 3), np.float32), normal=n,
                            light_dir=np.float32([0.0, 0.0, 1.0]), shade_mode=S.SHADE_LAMBERT))
    ds = [DeviceScene.from_host(s) for s in host]
    r = Rasterizer(64, 32)
    fbs = r.forward_batch(ds)
    gs = []
    for s in host:
        g = torch.zeros((s.height, s.width, 4), device="cuda")
        g[..., 0] = 1.0
        gs.append(g)
    for _ in range(2):  # the sums are left clear for the next call
        dls = [torch.zeros(3, device="cuda") for _ in host]
        dcs = [torch.zeros_like(d.color) for d in ds]
        r.backward_batch(ds, fbs, gs, dcs, None, dls)
        for s, dl, dc in zip(host, dls, dcs):
            T = s.num_triangles
            want = T * s.normal[0].astype(np.float64)
            # at most T additions, of which one rounding each
            assert (np.abs(dl.cpu().numpy() - want) <= T * 2.0 ** -25 * want).all()
            dc = dc.cpu().numpy()
            assert np.array_equal(dc[s.tris][:, :, 0], np.tile(np.float32([0.25, 0.25, 0.5]), (T, 1)))
            assert dc.sum(dtype=np.float64) == T
    r.close()


def test_colour_sums_of_a_vertex_of_many_pixels():
    """A vertex that takes the same sum r from each of 8,192 rows (one column of a
    triangle whose weight is constant along it): 8,192 r to within one rounding
    (half of 2^-24 on average) for each of 512 additions to one of 16 copies and of
    the 16 that join them.  2,048 additions to a copy are off by 1.9e-5 to 2.2e-5."""
    torch = _torch()
    from paper_1404_6293_gb300.raster import DeviceScene, Rasterizer
    W, H = 32, 8192
    px = np.array([(-20000.0, 4096.0), (100.0, -5000.0), (100.0, 13192.0)])
    pos = np.tile(np.float32([0, 0, 0, 1]), (300, 1))  # (the other vertices are unused)
    pos[:3, 0], pos[:3, 1] = px[:, 0] * (2.0 / W) - 1.0, 1.0 - px[:, 1] * (2.0 / H)
    s = S.Scene(W, H, pos, np.array([[0, 1, 2]], np.int32), color=np.ones((300, 3), np.float32))
    ds, r = DeviceScene.from_host(s), Rasterizer(W, H)
    fb = r.forward(ds)
    torch.cuda.synchronize()
    assert bool((fb.key != EMPTY).all())

    def sum_of(rows, x):
        g = torch.zeros((H, W, 4), device="cuda")
        g[:rows, x, 0] = 1.0
        return float(r.gradients(ds, fb, g, normal=False, light=False)[0][0, 0])

    for x in (3, 9, 15, 21):
        one = sum_of(1, x)
        assert abs(one - (99.5 - x) / 20100.0) <= 1e-6
        assert abs(sum_of(H, x) - H * one) <= 528 * 2.0 ** -25 * H * one
    r.close()


@pytest.mark.parametrize("size,bins", [((131, 137), 8), ((150, 70), 64), ((700, 300), 16), ((1200, 700), 32)])
def test_boxes_at_the_limits_on_the_direct_route(size, bins):
    """Boxes of 31 to 33 samples and 128 pixels, as many as the direct route asks
    for in small, medium and large frames."""
    from test_gpu_direct_raster import _LIMITS, _check, _triangles
    from paper_1404_6293_gb300 import _lib as L
    W, H = size
    copies = -(-W * H // (2 * len(_LIMITS))) + 1
    s = _triangles(W, H, _LIMITS, 5 * bins + W, copies)
    assert L.load().piko_raster_direct_scene(W, H, s.num_triangles, s.num_vertices) == 1
    _check(s, bins, "dynamic").close()


def test_meshes_on_both_sides_of_the_direct_lines():
    """Heightfields one step of tessellation apart around each line."""
    from test_gpu_direct_raster import _check
    from paper_1404_6293_gb300 import _lib as L
    for W, H, line in ((301, 211, 4), (640, 400, 7), (1100, 800, 10)):
        taken = []
        for px in (line * 0.9, line * 1.1):
            q = int((W * H / px / 2) ** 0.5)
            s = S.heightfield(W, H, q, q, seed=q, with_color=True)
            taken.append(L.load().piko_raster_direct_scene(W, H, s.num_triangles, s.num_vertices))
            _check(s, 16, "static").close()
        assert taken == [1, 0]
