"""Timed workloads of the rasterizer: the calls a renderer, a deferred-shading
engine, a Reyes sampler and a differentiable-rendering training loop make
through the public Python API, with their inputs, their algorithmic bytes and
a float64 statement of their results.

A case is a dict of plain values:
  kind       frame     one scene: Rasterizer.forward (and deferred_light for a G-buffer case)
             host      one scene in pinned host memory: Rasterizer.forward_host
             grad      one scene's gradients under a fixed framebuffer: Rasterizer.backward
             render    autograd.render and its backward, one view
             views     forward_batch + backward_batch of many views of one mesh
             batch     forward_batch + backward_batch of scenes of uneven size
  scene      random | heightfield | powerlaw | reyes | sphere (the generators of scenes.py)
  and the scene's sizes, the handle's bin size and schedule, and its options.
"""
import dataclasses
import math
import random as _random

import numpy as np
import torch

from paper_1404_6293_gb300 import _lib as L
from paper_1404_6293_gb300 import scenes as S
from paper_1404_6293_gb300.autograd import render
from paper_1404_6293_gb300.raster import DeviceScene, Framebuffer, HostScene, Rasterizer

_EMPTY = -1  # the all-ones key of an empty pixel, as int64


def listed():
    """What each stands for is said beside it."""
    return [
        # a small interactive view or thumbnail with the library's defaults: launches and the host decide
        dict(name="frame-256-defaults", kind="frame", scene="random", width=256, height=256, tris=1000, radius=40.0,
             bins=16, schedule="static", check=1),
        # a dense terrain at full HD, the benchmark's own frame: triangles of about two pixels
        dict(name="frame-1080p-terrain", kind="frame", scene="heightfield", width=1920, height=1080, nx=1000, ny=500,
             bins=32, schedule="hardware", check=0),
        # a terrain of ordinary size in a window of an odd size: perspective-correct attributes with
        # colours, the capacity check left on, the work-queue schedule
        dict(name="frame-odd-terrain", kind="frame", scene="heightfield", width=1283, height=717, nx=317, ny=211,
             color=1, persp=1, bins=16, schedule="dynamic", check=1),
        # the camera inside the scene: triangles cross the near and far planes and are clipped
        dict(name="frame-flythrough-clip", kind="frame", scene="heightfield", width=1280, height=720, nx=400, ny=300,
             color=1, persp=1, clip=1, bins=16, schedule="static", check=1),
        # deferred shading: G-buffer of triangles from one pixel to a quarter of the screen, then 64 lights
        dict(name="gbuffer-1080p-64-lights", kind="frame", scene="powerlaw", width=1920, height=1080, tris=500000,
             lights=64, bins=16, schedule="hardware", check=0),
        # Reyes sampling: micropolygon grids of half-pixel quads
        dict(name="frame-micropolygons", kind="frame", scene="reyes", width=1024, height=768, patches=256, bins=32,
             schedule="dynamic", check=0),
        # a large offline frame with the library's defaults
        dict(name="frame-4k-terrain", kind="frame", scene="heightfield", width=3840, height=2160, nx=2000, ny=1000,
             color=1, bins=16, schedule="static", check=1),
        # host memory in, host memory out: the end-to-end frame of a program that keeps its scene on the host
        dict(name="host-1080p-terrain", kind="host", scene="heightfield", width=1920, height=1080, nx=1000, ny=500,
             bins=32, schedule="hardware", check=1),
        # gradients of a dense frame (colours, normals and light), visibility fixed
        dict(name="grad-1080p-terrain", kind="grad", scene="heightfield", width=1920, height=1080, nx=1000, ny=500,
             color=1, bins=32, schedule="hardware", check=0),
        # one step of fitting an object from one view, through torch autograd
        dict(name="render-512-sphere", kind="render", scene="sphere", width=512, height=512, slices=250, stacks=200,
             bins=16, schedule="static", check=1),
        # one step of fitting an object from 64 views at once
        dict(name="views-64-sphere", kind="views", scene="sphere", width=512, height=512, slices=250, stacks=200,
             views=64, bins=16, schedule="dynamic", check=0),
        # a training batch of scenes of uneven sizes and kinds
        dict(name="batch-64-scenes", kind="batch", scenes=64, tmin=1000, tmax=200000, smin=256, smax=1024, bins=32,
             schedule="dynamic", check=0),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _bins(rng):
    return dict(bins=rng.choice([8, 16, 16, 16, 32, 32, 64]), schedule=rng.choice(["static", "dynamic", "hardware"]))


def draw(rng):
    """One case of the same ranges, sizes spread evenly over their logarithm."""
    kind = rng.choice(["random", "heightfield", "heightfield", "powerlaw", "reyes", "host", "grad", "render", "views",
                       "batch"])
    width = int(_log(rng, 96, 2560))
    height = max(48, int(width * rng.uniform(0.4, 1.0)))
    size = dict(width=width, height=height, check=rng.choice([0, 1]), **_bins(rng))
    if kind == "random":
        tris = int(_log(rng, 200, 100000))
        radius = min(64.0, max(2.0, math.sqrt(rng.uniform(1.0, 8.0) * width * height / tris)))
        return dict(kind="frame", scene="random", tris=tris, radius=round(radius, 2), mode=rng.choice([0, 1]), **size)
    if kind in ("heightfield", "host", "grad"):
        nx = int(_log(rng, 40, 1000))
        ny = max(10, int(nx * rng.uniform(0.4, 0.8)))
        c = dict(kind={"heightfield": "frame"}.get(kind, kind), scene="heightfield", nx=nx, ny=ny,
                 color=1 if kind == "grad" else rng.choice([0, 1]), persp=rng.choice([0, 1]), **size)
        if kind == "heightfield" and rng.random() < 0.3:
            c.update(clip=1, color=1)
        return c
    if kind == "powerlaw":
        return dict(kind="frame", scene="powerlaw", tris=int(_log(rng, 1000, 500000)),
                    lights=int(_log(rng, 1, 128)), exact_bins=rng.choice([0, 0, 1]), **size)
    if kind == "reyes":
        size.update(width=min(width, 1280), height=min(height, 1024))
        return dict(kind="frame", scene="reyes", patches=int(_log(rng, 4, 256)), **size)
    slices = int(_log(rng, 24, 250))
    side = int(_log(rng, 64, 640))
    size.update(width=side, height=max(48, int(side * rng.uniform(0.6, 1.0))))
    if kind in ("render", "views"):
        c = dict(kind=kind, scene="sphere", slices=slices, stacks=max(12, int(slices * 0.8)), persp=rng.choice([0, 1]),
                 **size)
        if kind == "views":
            c["views"] = int(_log(rng, 2, 48))
        return c
    return dict(kind="batch", scenes=int(_log(rng, 3, 48)), tmin=int(_log(rng, 200, 2000)),
                tmax=int(_log(rng, 5000, 200000)), smin=128, smax=int(_log(rng, 192, 1024)), check=size["check"],
                **_bins(rng))


# ------------------------------------------------------------------ scenes
def _batch_sizes(case):
    """(generator, triangles, width, height) per scene: triangle counts spread
    over their logarithm, sides over their range, in a mixed order."""
    n, out = case["scenes"], []
    for k in range(n):
        t = case["tmin"] * (case["tmax"] / case["tmin"]) ** (((7 * k) % n + 0.5) / n)
        side = int(case["smin"] + (case["smax"] - case["smin"]) * (((5 * k) % n + 0.5) / n))
        out.append(("random" if k % 2 else "heightfield", int(round(t)), side, max(64, side - 3 * (k % 11))))
    return out


def _flythrough(scene, seed):
    """A camera low over the terrain, looking along it: the near plane cuts the
    ground under the eye and the far plane the distance."""
    rng = _random.Random(seed)
    zs = float(scene.pos[:, 2].max())
    eye = [rng.uniform(-0.2, 0.2), rng.uniform(0.16, 0.2), 0.7 * zs]
    mvp = S._look_at_perspective(eye, [rng.uniform(-0.3, 0.3), -0.1, -zs], [0.0, 1.0, 0.0], 70.0,
                                 scene.width / scene.height, 0.3 * zs, 1.5 * zs)
    return dataclasses.replace(scene, mvp=mvp.astype(np.float32).ravel())


def _host_scenes(case, seed):
    """The case's scenes as numpy arrays (one, or the batch's)."""
    w, h = case.get("width"), case.get("height")
    kind = case.get("scene")
    if case["kind"] == "batch":
        out = []
        for k, (gen, t, bw, bh) in enumerate(_batch_sizes(case)):
            if gen == "random":
                radius = float(np.clip(np.sqrt(3.0 * bw * bh / t / 0.2321), 2.0, 64.0))
                out.append(S.random_triangles(bw, bh, t, radius, seed=seed * 1009 + k, shade_mode=S.SHADE_LAMBERT,
                                              with_normals=True))
            else:
                q = max(1, int(round(math.sqrt(t / 2.0))))
                out.append(S.heightfield(bw, bh, q, max(1, t // (2 * q)), seed=seed * 1009 + k, with_color=True))
        return out
    if kind == "random":
        return [S.random_triangles(w, h, case["tris"], case["radius"], seed=seed, shade_mode=case.get("mode", 0))]
    if kind == "heightfield":
        s = S.heightfield(w, h, case["nx"], case["ny"], seed=seed, with_color=bool(case.get("color")))
        return [_flythrough(s, seed) if case.get("clip") else s]
    if kind == "powerlaw":
        return [S.power_law_triangles(w, h, case["tris"], seed=seed)]
    if kind == "reyes":
        return [S.reyes_grids(w, h, case["patches"], seed=seed)]
    s, mvps = S.sphere_views(case.get("views", 1), w, h, case["slices"], case["stacks"], seed=seed)
    return [dataclasses.replace(s, mvp=m) for m in mvps]


def _handle(case, width, height):
    r = Rasterizer(width, height, case["bins"], case["bins"], case["schedule"])
    for name, opt in (("persp", L.PIKO_OPT_PERSPECTIVE), ("clip", L.PIKO_OPT_CLIP),
                      ("exact_bins", L.PIKO_OPT_EXACT_BINS)):
        if case.get(name):
            r.set_option(opt, 1)
    return r


def _fixed_sizes(case, r, first_pass):
    """A program that turns the capacity check off has sized its handle with
    one checked pass before."""
    if not case["check"]:
        first_pass()
        torch.cuda.synchronize()
        r.set_option(L.PIKO_OPT_CHECK_CAPACITY, 0)


def _flat_frames(sizes):
    """Framebuffers of all scenes in two tensors, and views of each scene's."""
    offs = np.concatenate([[0], np.cumsum([w * h for w, h in sizes])])
    key = torch.empty(int(offs[-1]), dtype=torch.int64, device="cuda")
    rgba = torch.empty((int(offs[-1]), 4), dtype=torch.float32, device="cuda")
    fbs = [Framebuffer(key[a:b].view(h, w), rgba[a:b].view(h, w, 4))
           for (w, h), a, b in zip(sizes, offs[:-1], offs[1:])]
    return key, rgba, fbs, offs


def _upstream(shape, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.randn(shape, generator=g, device="cuda", dtype=torch.float32)


def prepare(case, seed):
    kind = case["kind"]
    hosts = _host_scenes(case, seed)
    st = {"case": case}
    if kind in ("views", "batch"):
        if kind == "views":
            base = DeviceScene.from_host(hosts[0])
            mv = torch.from_numpy(np.stack([h.mvp for h in hosts])).cuda()
            scenes = [dataclasses.replace(base, mvp=mv[v]) for v in range(len(hosts))]
            c, n, l = (torch.zeros_like(t) for t in (base.color, base.normal, base.light_dir))
            st["grads"] = (c, n, l)
            st["gviews"] = ([c] * len(hosts), [n] * len(hosts), [l] * len(hosts))
        else:
            scenes = [DeviceScene.from_host(s) for s in hosts]
            vs = [s.num_vertices for s in hosts]
            c, n = (torch.zeros((sum(vs), 3), device="cuda") for _ in range(2))
            l = torch.zeros((len(hosts), 3), device="cuda")
            st["grads"] = (c, n, l)
            st["gviews"] = (list(c.split(vs)), list(n.split(vs)), [l[k] for k in range(len(hosts))])
        key, rgba, fbs, offs = _flat_frames([(s.width, s.height) for s in hosts])
        g = _upstream(rgba.shape, seed)
        r = _handle(case, hosts[0].width, hosts[0].height)
        knobs = ([(case["bins"],) * 2] * len(hosts), [case["schedule"]] * len(hosts))
        st.update(r=r, scenes=scenes, fbs=fbs, key=key, rgba=rgba, knobs=knobs,
                  gl=[g[a:b].view(s.height, s.width, 4) for s, a, b in zip(hosts, offs[:-1], offs[1:])])
        _fixed_sizes(case, r, lambda: r.forward_batch(scenes, fbs, *knobs))
        return st
    s = hosts[0]
    st["r"] = r = _handle(case, s.width, s.height)
    if kind == "host":
        hs = HostScene.from_host(s)
        fb = Framebuffer(torch.empty((s.height, s.width), dtype=torch.int64).pin_memory(),
                         torch.empty((s.height, s.width, 4)).pin_memory())
        st.update(scene=hs, fb=fb)
        _fixed_sizes(case, r, lambda: r.forward_host(hs, fb))
        return st
    ds = DeviceScene.from_host(s)
    st["scene"] = ds
    if kind == "render":
        st["leaves"] = [t.clone().requires_grad_(True) for t in (ds.color, ds.normal, ds.light_dir)]
        st["g"] = _upstream((s.height, s.width, 4), seed)
        _fixed_sizes(case, r, lambda: r.forward(ds))
        return st
    fb = Framebuffer.allocate(s.width, s.height, s.shade_mode)
    st["fb"] = fb
    if kind == "grad":
        r.forward(ds, fb)
        torch.cuda.synchronize()
        st["g"] = _upstream((s.height, s.width, 4), seed)
        st["grads"] = tuple(torch.zeros_like(t) for t in (ds.color, ds.normal, ds.light_dir))
        return st
    if case.get("lights"):
        st["lights"] = torch.from_numpy(S.point_lights(s.width, s.height, case["lights"], seed=seed)).cuda()
        st["lit"] = torch.empty((s.height, s.width, 4), device="cuda")
    _fixed_sizes(case, r, lambda: r.forward(ds, fb))
    return st


def run(st):
    kind, r = st["case"]["kind"], st["r"]
    if kind in ("views", "batch"):
        r.forward_batch(st["scenes"], st["fbs"], *st["knobs"])
        for t in st["grads"]:
            t.zero_()
        r.backward_batch(st["scenes"], st["fbs"], st["gl"], *st["gviews"])
        return [st["key"], st["rgba"], *st["grads"]]
    if kind == "host":
        # the results are in host memory once the stream has passed the call: a program waits for them
        fb = r.forward_host(st["scene"], st["fb"])
        torch.cuda.current_stream().synchronize()
        return [fb.key, fb.rgba]
    if kind == "render":
        rgba, key = render(r, st["scene"], *st["leaves"])
        return [key, rgba, *torch.autograd.grad(rgba, st["leaves"], st["g"])]
    if kind == "grad":
        for t in st["grads"]:
            t.zero_()
        return list(r.backward(st["scene"], st["fb"], st["g"], *st["grads"]))
    fb = r.forward(st["scene"], st["fb"])
    if "lights" in st:
        return [fb.key, fb.gbuf_normal, fb.gbuf_albedo, r.deferred_light(fb, st["lights"], st["lit"])]
    return [fb.key, fb.rgba]


# -------------------------------------------------------------------- work
def _counts(case):
    """(vertices, triangles, pixels, colours, normals) per scene."""
    w, h = case.get("width"), case.get("height")
    if case["kind"] == "batch":
        out = []
        for gen, t, bw, bh in _batch_sizes(case):
            if gen == "random":
                out.append((3 * t, t, bw * bh, 1, 1))
            else:
                q = max(1, int(round(math.sqrt(t / 2.0))))
                p = max(1, t // (2 * q))
                out.append(((q + 1) * (p + 1), 2 * q * p, bw * bh, 1, 1))
        return out
    kind = case["scene"]
    if kind == "random":
        return [(3 * case["tris"], case["tris"], w * h, 1, case.get("mode", 0))]
    if kind == "heightfield":
        nx, ny = case["nx"], case["ny"]
        return [((nx + 1) * (ny + 1), 2 * nx * ny, w * h, case.get("color", 0), 1)]
    if kind == "powerlaw":
        return [(3 * case["tris"], case["tris"], w * h, 1, 1)]
    if kind == "reyes":  # a patch of log-uniform side in [16, 160] px, diced to half-pixel quads, 128 at most: 9,855 on average
        t = int(2 * 9855 * case["patches"])
        return [(t // 2, t, w * h, 1, 1)]
    sl, stk = case["slices"], case["stacks"]
    return [((stk - 1) * sl + 2, 2 * sl * (stk - 1), w * h, 1, 1)] * case.get("views", 1)


def work(case):
    """Forward: positions, attributes and indices in, 8-byte keys and 16 bytes
    of colour (or G-buffer) out.  Gradients: keys, dL/drgba, indices, positions
    and attributes in, one array of sums out per attribute.  The light pass:
    the G-buffer in, colours out, about 20 operations per pixel and light."""
    counts = _counts(case)
    kind = case["kind"]
    many = len(counts) > 1 and kind == "views"
    fwd = bwd = 0
    for k, (v, t, p, c, n) in enumerate(counts):
        first = not many or k == 0  # the views share one mesh
        geo = (16 * v + 12 * t + 12 * v * (c + n)) if first else 0
        fwd += geo + 24 * p
        bwd += geo + 24 * p + (12 * v * (c + n) if first else 0)
    flops = 0
    if case.get("lights"):
        p = counts[0][2]
        fwd += (24 + 16) * p
        flops = 20 * p * case["lights"]
    if kind == "grad":
        return {"bytes": bwd, "flops": 0}
    if kind in ("render", "views", "batch"):
        return {"bytes": fwd + bwd, "flops": 0}
    return {"bytes": fwd, "flops": flops}


# ------------------------------------------------------------------- exact
# The results in 64 bits from plain torch: the definition's float32 transform
# and 16.8 snap, then integer edge functions, fill rule and depth, and the
# shading, lighting and gradients in float64.
def _clip_space(pos, mvp):
    if mvp is None:
        return [pos[:, q] for q in range(4)]
    m = mvp.reshape(4, 4)
    rows = []
    for q in range(4):
        acc = m[q, 0] * pos[:, 0]
        for j in range(1, 4):
            acc = acc + m[q, j] * pos[:, j]
        rows.append(acc)
    return rows


def _viewport(x, y, z, w, W, H):
    nx, ny, nz = x / w, y / w, z / w
    fx = ((nx * 0.5 + 0.5) * float(W)) * 256.0
    fy = ((0.5 - ny * 0.5) * float(H)) * 256.0
    sz = (nz * 0.5 + 0.5) * 16777215.0
    inside = (fx.abs() < 8388608.0) & (fy.abs() < 8388608.0)
    return nz, fx, fy, sz, inside


def _ints(ok, *fs):
    return [torch.where(ok, torch.round(f), torch.zeros_like(f)).to(torch.int64) for f in fs]


def _plane(pts, n, near):
    """One Sutherland-Hodgman pass over polygons pts [N,8,4] with n corners."""
    out, m = torch.zeros_like(pts), torch.zeros_like(n)
    rows = torch.arange(len(n), device=n.device)
    for k in range(8):
        live = k < n
        a, b = pts[:, k], pts[rows, torch.where(k + 1 < n, torch.full_like(n, k + 1), torch.zeros_like(n)).clamp(max=7)]
        da, db = (a[:, 2] + a[:, 3], b[:, 2] + b[:, 3]) if near else (a[:, 3] - a[:, 2], b[:, 3] - b[:, 2])
        ina, inb = da >= 0, db >= 0
        keep = live & ina
        out[rows[keep], m[keep]] = a[keep]
        m = m + keep
        cut = live & (ina != inb)
        t = (da / (da - db))[:, None]
        v = a + t * (b - a)
        out[rows[cut], m[cut]] = v[cut]
        m = m + cut
    return out, m


def _points(pos, tris, mvp, W, H, clip):
    """Snapped points [N,3] of X, Y, Z, the triangle of each, and which triangles were clipped."""
    c = _clip_space(pos, mvp)
    nz, fx, fy, sz, inside = _viewport(*c, W, H)
    ok = (c[3] > 0) & (nz >= -1) & (nz <= 1) & inside
    X, Y, Z = _ints(ok, fx, fy, sz)
    good = ok[tris].all(1)
    ids = good.nonzero()[:, 0]
    P = [q[tris[ids]] for q in (X, Y, Z)]
    if clip and not bool(good.all()):
        bad = (~good).nonzero()[:, 0]
        pts = torch.zeros((len(bad), 8, 4), device=pos.device)
        pts[:, :3] = torch.stack(c, 1)[tris[bad]]
        n = torch.full((len(bad),), 3, device=pos.device)
        pts, n = _plane(pts, n, True)
        pts, n = _plane(pts, n, False)
        w = pts[..., 3]
        _, fx, fy, sz, inside = _viewport(*(pts[..., q] for q in range(4)), W, H)
        okp = (w > 0) & inside
        sz = torch.nan_to_num(torch.round(sz), nan=0.0).clamp(0.0, 16777215.0)
        X, Y, Z = _ints(okp, fx, fy, sz)
        for k in range(1, 7):
            use = (k + 1 < n) & okp[:, 0] & okp[:, k] & okp[:, k + 1]
            sel = torch.tensor([0, k, k + 1], device=pos.device)
            P = [torch.cat([p, q[use][:, sel]]) for p, q in zip(P, (X, Y, Z))]
            ids = torch.cat([ids, bad[use]])
    return P, ids, good


def _visible(P, ids, W, H):
    """The key of every pixel (int64, the largest value where empty)."""
    X, Y, Z = P
    far = torch.iinfo(torch.int64).max
    key = torch.full((W * H,), far, dtype=torch.int64, device=X.device)
    A = (X[:, 1] - X[:, 0]) * (Y[:, 2] - Y[:, 0]) - (X[:, 2] - X[:, 0]) * (Y[:, 1] - Y[:, 0])
    flip = torch.where((A < 0)[:, None], torch.tensor([0, 2, 1], device=X.device), torch.tensor([0, 1, 2], device=X.device))
    X, Y, Z, A = X.gather(1, flip), Y.gather(1, flip), Z.gather(1, flip), A.abs()
    x0 = ((X.amin(1) + 127) >> 8).clamp(min=0)
    x1 = ((X.amax(1) - 128) >> 8).clamp(max=W - 1)
    y0 = ((Y.amin(1) + 127) >> 8).clamp(min=0)
    y1 = ((Y.amax(1) - 128) >> 8).clamp(max=H - 1)
    bw, bh = (x1 - x0 + 1).clamp(min=0), (y1 - y0 + 1).clamp(min=0)
    live = ((bw * bh > 0) & (A > 0)).nonzero()[:, 0]
    if len(live) == 0:
        return key
    cnt = (bw * bh)[live]
    ends = cnt.cumsum(0)
    total, lo = int(ends[-1]), 0
    while lo < len(live):
        start = int(ends[lo - 1]) if lo else 0
        hi = max(lo + 1, int(torch.searchsorted(ends, torch.tensor(start + (1 << 23), device=ends.device))))
        sub, n = live[lo:hi], cnt[lo:hi]
        own = torch.repeat_interleave(sub, n)
        k = torch.arange(len(own), device=X.device) - torch.repeat_interleave(ends[lo:hi] - n - start, n)
        yy = k // bw[own]
        px, py = x0[own] + k - yy * bw[own], y0[own] + yy
        cx, cy = 256 * px + 128, 256 * py + 128
        w, cov = [], torch.ones_like(px, dtype=torch.bool)
        for i, j in ((1, 2), (2, 0), (0, 1)):
            dx, dy = (X[:, j] - X[:, i])[own], (Y[:, j] - Y[:, i])[own]
            e = dx * (cy - Y[own, i]) - dy * (cx - X[own, i])
            top_left = (dy < 0) | ((dy == 0) & (dx > 0))
            cov &= e - (~top_left).to(e.dtype) >= 0
            w.append(e)
        own, px, py = own[cov], px[cov], py[cov]
        num = w[1][cov] * (Z[:, 1] - Z[:, 0])[own] + w[2][cov] * (Z[:, 2] - Z[:, 0])[own]
        z = Z[own, 0] + torch.div(num, A[own], rounding_mode="floor")
        key.scatter_reduce_(0, py * W + px, (z << 32) | ids[own], "amin")
        lo = hi
    return key


def _winners(s, clip, persp):
    """Covered pixels, their key, their triangle's vertices and float64 weights."""
    W, H = s["W"], s["H"]
    P, ids, good = _points(s["pos"], s["tris"], s["mvp"], W, H, clip)
    key = _visible(P, ids, W, H)
    full = key != torch.iinfo(torch.int64).max
    pix = full.nonzero()[:, 0]
    t = key[pix] & 0xFFFFFFFF
    v = s["tris"][t]
    x, y = pix % W, pix // W
    c = _clip_space(s["pos"], s["mvp"])
    nz, fx, fy, sz, inside = _viewport(*c, W, H)
    X, Y = _ints((c[3] > 0) & inside, fx, fy)
    X, Y = X[v], Y[v]
    cx, cy = (256 * x + 128)[:, None], (256 * y + 128)[:, None]
    i, j = [1, 2, 0], [2, 0, 1]
    e = (X[:, j] - X[:, i]) * (cy - Y[:, i]) - (Y[:, j] - Y[:, i]) * (cx - X[:, i])
    b = e.double() / e.sum(1, keepdim=True).double()
    cw = c[3][v].double()
    if persp:
        q = b / cw
        b = q / q.sum(1, keepdim=True)
    if clip:  # a clipped triangle's weights at the pixel centre's ray
        xn, yn = ((x.double() + 0.5) / W) * 2 - 1, 1 - ((y.double() + 0.5) / H) * 2
        a = c[0][v].double() - xn[:, None] * cw
        d = c[1][v].double() - yn[:, None] * cw
        q = torch.stack([a[:, i[k]] * d[:, j[k]] - a[:, j[k]] * d[:, i[k]] for k in range(3)], 1)
        b = torch.where(good[t][:, None], b, q / q.sum(1, keepdim=True))
    return torch.where(full, key, torch.full_like(key, _EMPTY)), pix, t, v, b


def _mix(b, attr, v):
    return (b[:, :, None] * attr[v].double()).sum(1)


def _albedo(s, v, b):
    if s["color"] is not None:
        return _mix(b, s["color"], v)
    return torch.tensor([0.80, 0.75, 0.65], dtype=torch.float32, device=b.device).double().expand(len(b), 3)


def _image(s, pix, rgb):
    out = torch.zeros((s["W"] * s["H"], 4), dtype=torch.float64, device=rgb.device)
    out[pix, :3] = rgb
    out[pix, 3] = 1.0
    return out


def _shaded(s, clip, persp, lights=None):
    key, pix, t, v, b = _winners(s, clip, persp)
    rgb = _albedo(s, v, b)
    nrm = _mix(b, s["normal"], v) if s["normal"] is not None else None
    if s["mode"] == S.SHADE_LAMBERT:
        rgb = rgb * (nrm @ s["light"].double()).clamp(min=0)[:, None]
    W, H = s["W"], s["H"]
    if s["mode"] != S.SHADE_GBUFFER:
        return [key.view(H, W), _image(s, pix, rgb).view(H, W, 4)], (pix, v, b, nrm)
    n4 = torch.zeros((W * H, 4), dtype=torch.float64, device=b.device)
    n4[pix, :3] = nrm
    # the light pass reads the binary16 G-buffer
    n, a = nrm.half().double(), rgb.half().double()
    D = float(max(W, H))
    p = torch.stack([pix % W + 0.5, pix // W + 0.5, (key[pix] >> 32) / 16777215.0 * D], 1).double()
    acc = torch.zeros(len(pix), dtype=torch.float64, device=b.device)
    for lx in lights.double():
        d = lx[:3] - p
        d2 = (d * d).sum(1)
        lam = ((n * d).sum(1) / d2.sqrt()).clamp(min=0)
        acc += torch.where(d2 > 0, lx[3] * lam / (1 + d2 / (D / 4) ** 2), torch.zeros_like(acc))
    return [key.view(H, W), n4.view(H, W, 4), _image(s, pix, rgb).view(H, W, 4),
            _image(s, pix, a * acc[:, None]).view(H, W, 4)], None


def _gradients(s, won, g, out=None):
    """Adds dL/dcolour, dL/dnormal and dL/dlight of one scene to out."""
    pix, v, b, nrm = won
    dc, dn, dl = out or [torch.zeros_like(s[k], dtype=torch.float64) for k in ("color", "normal", "light")]
    g = g.reshape(-1, 4)[pix, :3].double()
    Lt = s["light"].double()
    d = nrm @ Lt
    alb = _albedo(s, v, b)
    G = torch.where(d > 0, (g * alb).sum(1), torch.zeros_like(d))
    for k in range(3):
        dc.index_add_(0, v[:, k], g * (d.clamp(min=0) * b[:, k])[:, None])
        dn.index_add_(0, v[:, k], (G * b[:, k])[:, None] * Lt)
    dl += (G[:, None] * nrm).sum(0)
    return dc, dn, dl


def _plain(h):
    def t(a, dt=torch.float32):
        return None if a is None else torch.from_numpy(np.ascontiguousarray(a)).to("cuda", dt)
    return {"W": h.width, "H": h.height, "pos": t(h.pos), "tris": t(h.tris, torch.int64), "color": t(h.color),
            "normal": t(h.normal), "mvp": t(h.mvp), "light": t(h.light_dir), "mode": h.shade_mode}


def exact(case, seed):
    kind, clip, persp = case["kind"], bool(case.get("clip")), bool(case.get("persp"))
    hosts = _host_scenes(case, seed)
    if kind in ("views", "batch"):
        shape = (sum(h.width * h.height for h in hosts), 4)
        g, at, keys, imgs, outs = _upstream(shape, seed), 0, [], [], []
        sums = None
        for h in hosts:
            s = _plain(h)
            (key, img), won = _shaded(s, clip, persp)
            n = h.width * h.height
            got = _gradients(s, won, g[at:at + n], sums)
            if kind == "views":
                sums = got
            else:
                outs.append(got)
            keys.append(key.reshape(-1))
            imgs.append(img.reshape(-1, 4))
            at += n
        if kind == "batch":
            sums = [torch.cat([o[0] for o in outs]), torch.cat([o[1] for o in outs]), torch.stack([o[2] for o in outs])]
        return [torch.cat(keys), torch.cat(imgs), *sums]
    s = _plain(hosts[0])
    lights = None
    if case.get("lights"):
        lights = torch.from_numpy(S.point_lights(s["W"], s["H"], case["lights"], seed=seed)).cuda()
    outs, won = _shaded(s, clip, persp, lights)
    if kind in ("frame", "host"):
        return outs
    grads = _gradients(s, won, _upstream((s["H"], s["W"], 4), seed))
    return list(grads) if kind == "grad" else [*outs, *grads]
