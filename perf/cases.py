"""Performance cases of the ray caster: what a viewer, a fitting loop and a server have it do.

``listed()`` gives the cases that are timed, ``draw(rng)`` one more of the same ranges,
``prepare(case, seed)`` what a program holds before the call (inputs on the GPU, a context, a
loaded and bricked cube), ``run(state)`` one pass through the package's public calls,
``work(case)`` the bytes and operations a pass cannot do without, and ``exact(case, seed)`` the
same outputs in 64 bits by plain torch and numpy.  Every case is a dict of plain values.

Kinds
  frame    a viewer's frames of a resident cube: a new camera, then the frame (device output)
  viewer   the same with host buffers: colour map, spectral-channel mask, render window and camera
           sent by the viewer, the frame copied back to pinned memory
  fit      a fitting step: views of the current voxels and table, an L2 loss against target
           images, gradients with respect to both
  ingest   new data: load, exact min/max, bricking, first frame, release
  compress new data kept compressed: load, wavelet compression, bricking, first frame, release
  serve    a batch of viewers' requests on two cubes through the request loop
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1008_0135_gb300 as vr
from paper_1008_0135_gb300.autograd import render_views

DEV = "cuda"


def _case(name, kind, **kw):
    base = dict(kind=kind, nx=64, ny=64, nz=64, brick=32, storage="f32", layouts=9, mode="dvr", term="segment",
                step=0.5, tau=0.99, proj="persp", W=256, H=256, views=1, elev=0.0, table="ramp", vmin=-3.0,
                vmax=20.0, data="sources", noise=1.0)
    base.update(kw)
    if name:
        base["name"] = name
    return base


def listed():
    hipass = dict(nx=1720, ny=1720, nz=1024, brick=256, step=1.0, W=1024, H=1024, vmin=-3.0, vmax=100.0)
    small = dict(hipass, nx=768, ny=768, nz=512)
    return [
        # the smallest frame, where launches and host work count: a 64^3 cube in 8 bricks
        _case("frame 64^3", "frame", proj="ortho"),
        # the headline: a HIPASS-scale cube (12 GB), perspective orbit, one view per pass
        _case("frame hipass f32", "frame", **hipass),
        # the same with FP16 bricks, how a viewer halves the cube's footprint
        _case("frame hipass f16", "frame", storage="f16", **hipass),
        # maximum-intensity projection, the other output of the viewer
        _case("mip 768x768x512", "frame", mode="mip", elev=15.0, **small),
        # opaque colour map with rays stopping globally (occlusion skipping)
        _case("opaque 768x768x512", "frame", term="global", table="opaque", elev=15.0, **small),
        # an all-sky survey slab at step 0.5 with BF16 bricks read through pair atlases
        _case("frame gass slab bf16", "frame", nx=2048, ny=2048, nz=256, brick=256, storage="bf16", layouts=41,
              W=1024, H=1024, vmin=-2.0, vmax=8.0, data="field", noise=0.5),
        # a viewer with host buffers on a ragged cube and frame, default (linear) brick layout,
        # every third channel off, a window
        _case("viewer 333x257x190", "viewer", nx=333, ny=257, nz=190, brick=100, layouts=1, W=641, H=479, elev=20.0),
        # fitting step of the differentiation workload: 256^3 voxels and table, 8 views at 512^2
        _case("fit 256^3", "fit", nx=256, ny=256, nz=256, brick=128, W=512, H=512, views=8),
        # a small fitting step, one view, only the table fitted
        _case("fit table 64^3", "fit", voxels=False),
        # a cube arrives (odd sizes): min/max, FP16 bricks with atlases, first frame
        _case("ingest 611x700x433", "ingest", nx=611, ny=700, nz=433, brick=128, storage="f16", W=1024, H=768,
              step=1.0, vmin=-3.0, vmax=100.0),
        # a cube arrives and is kept compressed; the first frame decodes its bricks
        _case("compress 768x768x512", "compress", **small),
        # twelve requests of several viewers, four in flight, frames of two cubes and both modes
        _case("serve 12", "serve", nx=512, ny=480, nz=384, brick=128, storage="f16", W=512, H=512, step=1.0,
              vmin=-3.0, vmax=100.0, requests=12),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["frame", "frame", "frame", "frame", "viewer", "fit", "fit", "ingest", "compress", "serve"])
    storage = rng.choice(["f32", "f32", "f16", "bf16"])
    wide = rng.random() < 0.5
    vmin, vmax = (-3.0, 100.0) if wide else (-3.0, 20.0)
    kw = dict(storage=storage, vmin=vmin, vmax=vmax, elev=round(rng.uniform(-40.0, 40.0), 2),
              step=rng.choice([0.5, 0.75, 1.0]), proj=rng.choice(["persp", "persp", "ortho"]),
              brick=rng.choice([48, 64, 100, 128, 256]))
    if kind == "frame":
        e = _log(rng, 64, 1200)
        kw.update(nx=_log(rng, max(40, e // 2), e * 5 // 4), ny=_log(rng, max(40, e // 2), e * 5 // 4),
                  nz=_log(rng, 40, e), W=_log(rng, 128, 1280), H=_log(rng, 128, 1024),
                  mode=rng.choice(["dvr", "dvr", "dvr", "mip"]), term=rng.choice(["segment", "segment", "global"]),
                  layouts=rng.choice([9, 9, 9, 41, 1, 7]), data=rng.choice(["sources", "field"]))
        kw["table"] = "opaque" if kw["term"] == "global" else "ramp"
    elif kind == "viewer":
        kw.update(nx=_log(rng, 60, 500), ny=_log(rng, 60, 500), nz=_log(rng, 60, 400), W=_log(rng, 200, 1280),
                  H=_log(rng, 200, 1024), layouts=rng.choice([1, 9]))
    elif kind == "fit":
        e = _log(rng, 48, 256)
        kw.update(storage="f32", nx=e, ny=max(40, e - rng.randrange(9)), nz=max(40, e - rng.randrange(9)),
                  W=_log(rng, 128, 512), H=_log(rng, 128, 512), views=rng.choice([1, 2, 3, 4, 8]),
                  layouts=rng.choice([1, 9, 9]), voxels=rng.random() < 0.7)
    elif kind == "ingest":
        kw.update(nx=_log(rng, 100, 768), ny=_log(rng, 100, 768), nz=_log(rng, 100, 512), W=_log(rng, 256, 1024),
                  H=_log(rng, 256, 1024), layouts=rng.choice([1, 9, 9]))
    elif kind == "compress":
        kw.update(storage="f32", nx=_log(rng, 100, 768), ny=_log(rng, 100, 768), nz=_log(rng, 100, 512),
                  W=_log(rng, 256, 1024), H=_log(rng, 256, 1024))
    else:
        kw.update(nx=_log(rng, 100, 512), ny=_log(rng, 100, 512), nz=_log(rng, 100, 384), W=_log(rng, 200, 700),
                  H=_log(rng, 200, 700), requests=rng.randrange(4, 13))
    if storage == "f32" or kind not in ("frame",):
        kw["layouts"] = 9 if kw.get("layouts") == 41 else kw.get("layouts", 9)
    if kind in ("fit", "compress"):
        kw["storage"] = "f32"
    return _case(None, kind, **kw)


# ------------------------------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) % (1 << 62))
    return g


def _cube(nx, ny, nz, data, noise, seed):
    """A spectral cube [z][y][x]: Gaussian noise, and either bar-like sources along the spectral
    axis with a faint band of emission (HIPASS-like) or a slab of large-scale structure (GASS-like)."""
    cube = torch.empty((nz, ny, nx), device=DEV)
    cube.normal_(0.0, noise, generator=_gen(seed))
    rng = np.random.default_rng(int(seed) + 17)
    z = torch.arange(nz, device=DEV) + 0.5
    if data == "field":
        lo, hi = nz // 8, nz - nz // 8
        f = torch.zeros((hi - lo, ny, nx), device=DEV)
        for o in range(3):
            c = 6 << o
            coarse = torch.randn((1, 1, 2 << o, c, c), device=DEV, generator=_gen(seed + 31 + o))
            f += torch.nn.functional.interpolate(coarse, size=f.shape, mode="trilinear", align_corners=True)[0, 0] * (2.0 * 0.35 ** o)
        cube[lo:hi] += f
        return cube
    n = int(min(192, max(8, nx * ny * nz / 3e5)))
    for _ in range(n):
        c = [rng.uniform(0, m) for m in (nx, ny, nz)]
        sxy = rng.uniform(1.0, 4.0) * max(1.0, min(nx, ny, nz) / 256)
        s = (sxy, sxy, sxy * rng.uniform(2.0, 5.0))
        amp = math.exp(rng.uniform(math.log(3.0), math.log(100.0)))
        sl, g = [], []
        for a, m in enumerate((nx, ny, nz)):
            i0, i1 = max(0, int(c[a] - 3 * s[a])), min(m, int(c[a] + 3 * s[a]) + 2)
            sl.append(slice(i0, i1))
            g.append(torch.exp(-((torch.arange(i0, i1, device=DEV) + 0.5 - c[a]) ** 2) / (2 * s[a] * s[a])))
        cube[sl[2], sl[1], sl[0]] += amp * g[2][:, None, None] * g[1][None, :, None] * g[0][None, None, :]
    cube += (2.0 * torch.exp(-((z - 0.5 * nz) ** 2) / (2 * 16.0 ** 2)))[:, None, None]
    return cube


def _case_cube(case, seed):
    return _cube(case["nx"], case["ny"], case["nz"], case["data"], case["noise"], seed)


def _table(kind, n=256):
    t = np.arange(n, dtype=np.float64) / (n - 1)
    return np.stack([t, t * t, 1.0 - t, t if kind == "opaque" else 0.1 * t], axis=1).astype(np.float32)


def _look(eye, target):
    f = np.asarray(target, np.float64) - np.asarray(eye, np.float64)
    f /= np.linalg.norm(f)
    r = np.cross(f, (0.0, 1.0, 0.0))
    r /= np.linalg.norm(r)
    m = np.eye(4)
    m[0, :3], m[1, :3], m[2, :3] = r, np.cross(r, f), -f
    m[:3, 3] = -m[:3, :3] @ np.asarray(eye, np.float64)
    return m.astype(np.float32)


def _cams(case, seed, n, W=None, H=None):
    """n views of an orbit about the y axis from a random azimuth."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    c = np.array([nx, ny, nz], np.float64) / 2
    half = 0.5 * math.sqrt(nx * nx + ny * ny + nz * nz)
    a0, el = np.random.default_rng(int(seed) + 5).uniform(0, 2 * math.pi), math.radians(case["elev"])
    out = []
    for j in range(n):
        a = a0 + 2 * math.pi * j / n
        d = np.array([math.sin(a) * math.cos(el), math.sin(el), math.cos(a) * math.cos(el)])
        ortho = case["proj"] == "ortho"
        out.append(dict(view=_look(c + (2.0 if ortho else 1.5) * half * d, c), proj=0 if ortho else 1,
                        param=2.0 * half if ortho else math.radians(60.0), W=W or case["W"], H=H or case["H"]))
    return out


def _mask(nz):
    m = np.ones(nz, np.uint8)
    m[::3] = 0
    return m


def _window(case):
    n = (case["nx"], case["ny"], case["nz"])
    return [m // 10 for m in n], [m - m // 12 for m in n]


def _targets(case, seed):
    """Target images of a fit: smooth premultiplied pictures."""
    g = torch.rand((case["views"], 4, 5, 5), device=DEV, generator=_gen(seed + 71))
    t = torch.nn.functional.interpolate(g, size=(case["H"], case["W"]), mode="bilinear", align_corners=True)
    return (0.5 * t).permute(0, 2, 3, 1).contiguous()


def _set_params(ctx, case):
    ctx.set_transfer_function(_table(case["table"]), case["vmin"], case["vmax"])
    ctx.set_render_params(case["mode"], case["step"], case["tau"])
    ctx.set_termination(case["term"])


def _requests(case, seed):
    """What the viewers of a serve case ask for: (cube 0 or 1, case of that cube, camera, mode, table)."""
    rng = np.random.default_rng(int(seed) + 9)
    out = []
    for i in range(case["requests"]):
        which = int(i % 3 == 2)
        sub = dict(case, **_second(case)) if which else case
        k = (1, 2, 1, 4)[i % 4]
        cam = _cams(dict(sub, elev=rng.uniform(-30, 30)), seed + 100 + i, 1, W=case["W"] * 2 // (k + 1), H=case["H"] * 2 // (k + 1))[0]
        out.append((which, sub, cam, "mip" if i % 5 == 4 else "dvr", "opaque" if i % 4 == 1 else "ramp"))
    return out


def _second(case):
    return dict(nx=case["nx"] // 2, ny=case["ny"] // 2, nz=case["nz"] // 2, storage="f32", step=0.5)


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case)
    cube = _case_cube(case, seed)
    if kind in ("ingest", "compress"):
        cache = 0
        if kind == "compress":
            b = [min(case["brick"], case[k]) + 2 for k in ("nx", "ny", "nz")]
            nb = [-(-case[k] // case["brick"]) for k in ("nx", "ny", "nz")]
            cache = (4 * b[0] * b[1] * b[2] + 256) * nb[0] * nb[1] * nb[2]
        st.update(ctx=vr.Context(0, cache_bytes=cache), cube=cube, cams=_cams(case, seed, 1))
        _set_params(st["ctx"], case)
        return st
    ctx = vr.Context(0)
    cid = ctx.load_cube(cube)
    ctx.set_brick_layouts(cid, case["layouts"])
    ctx.set_bricking(cid, (case["brick"],) * 3, 1, case["storage"])
    st.update(ctx=ctx, cid=cid)
    _set_params(ctx, case)
    if kind == "frame":
        st["cams"] = _cams(case, seed, case["views"])
    elif kind == "viewer":
        st.update(cams=_cams(case, seed, 1), table=_table(case["table"]), mask=_mask(case["nz"]),
                  host=torch.empty((case["H"], case["W"], 4)).pin_memory())
    elif kind == "fit":
        st.update(cams=_cams(case, seed, case["views"]), target=_targets(case, seed),
                  table=torch.from_numpy(_table(case["table"])).to(DEV),
                  voxels=cube if case.get("voxels", True) else None)
    elif kind == "serve":
        sub = _second(case)
        c2 = _cube(sub["nx"], sub["ny"], sub["nz"], case["data"], case["noise"], seed + 3)
        cid2 = ctx.load_cube(c2)
        ctx.set_brick_layouts(cid2, 9)
        ctx.set_bricking(cid2, (case["brick"],) * 3, 1, sub["storage"])
        reqs = []
        for which, sub, cam, mode, table in _requests(case, seed):
            shape = (cam["H"], cam["W"], 4) if mode == "dvr" else (cam["H"], cam["W"])
            reqs.append(dict(cube=cid2 if which else cid, cam=cam, mode=mode, step=sub["step"], tau=case["tau"],
                             lut=_table(table), vrange=(case["vmin"], case["vmax"]), arrival_ms=0.0,
                             out=torch.empty(shape, device=DEV)))
        st["reqs"] = reqs
    return st


# ------------------------------------------------------------------------------------- a pass
def run(st):
    case, ctx = st["case"], st["ctx"]
    kind = case["kind"]
    if kind == "frame":
        out = []
        for cam in st["cams"]:
            ctx.set_camera_dict(cam)
            out.append(ctx.render_frame(st["cid"]))
        return out
    if kind == "viewer":
        ctx.set_transfer_function(st["table"], case["vmin"], case["vmax"])
        ctx.set_channel_mask(st["mask"])
        ctx.set_window(*_window(case))
        ctx.set_camera_dict(st["cams"][0])
        return ctx.render_frame(st["cid"], out=st["host"])
    if kind == "fit":
        table = st["table"].detach().requires_grad_()
        vox = st["voxels"].detach().requires_grad_() if st["voxels"] is not None else None
        img = render_views(ctx, st["cid"], table, st["cams"], (case["vmin"], case["vmax"]), voxels=vox,
                           step=case["step"], tau=case["tau"])
        (0.5 * (img - st["target"]).square().sum()).backward()
        return {"img": img.detach(), "table": table.grad, "voxels": vox.grad if vox is not None else None}
    if kind == "ingest":
        cid = ctx.load_cube(st["cube"])
        lo, hi = ctx.compute_minmax(cid)
        ctx.set_brick_layouts(cid, case["layouts"])
        ctx.set_bricking(cid, (case["brick"],) * 3, 1, case["storage"])
        ctx.set_camera_dict(st["cams"][0])
        img = ctx.render_frame(cid)
        ctx.free_cube(cid)
        return {"range": np.array([lo, hi], np.float32), "img": img}
    if kind == "compress":
        cid = ctx.load_cube(st["cube"])
        ctx.compress_cube(cid)
        ctx.set_brick_layouts(cid, 9)
        ctx.set_bricking(cid, (case["brick"],) * 3, 1, "f32")
        ctx.set_camera_dict(st["cams"][0])
        img = ctx.render_frame(cid)
        ctx.free_cube(cid)
        return img
    res, _ = ctx.serve(st["reqs"], max_inflight=4)
    if any(r["status"] for r in res):
        raise RuntimeError("a request failed")
    return [r["out"] for r in st["reqs"]]


# ------------------------------------------------------------------------------------- work
def _samples(case, cam):
    """Samples of a frame: chords of a coarse grid of rays through the box, over the step, cut where the
    mean opacity of the noise would stop a ray (per brick or globally)."""
    with np.errstate(all="ignore"):
        lo, hi = (np.zeros(3), np.array([case["nx"], case["ny"], case["nz"]], np.float64))
        if case["kind"] == "viewer":
            w = _window(case)
            lo, hi = np.array(w[0], np.float64), np.array(w[1], np.float64)
        o, d = _rays(dict(cam, W=32, H=32), cam["W"] / cam["H"])
        t0, t1 = (lo - o) / d, (hi - o) / d
        chord = np.maximum(0.0, np.minimum(1e30, np.maximum(t0, t1)).min(1) - np.maximum(np.minimum(t0, t1).max(1), 0.0))
    n = chord / case["step"]
    if case["mode"] == "dvr":
        a = (0.0 - case["vmin"]) / (case["vmax"] - case["vmin"]) * (1.0 if case["table"] == "opaque" else 0.1)
        stop = math.log(1.0 / max(1e-6, 1 - case["tau"])) / a
        if case["term"] == "global":
            n = np.minimum(n, stop)
        else:
            n = n * min(1.0, stop / (case["brick"] / case["step"]))
    return float(n.mean()) * cam["W"] * cam["H"]


def work(case):
    kind = case["kind"]
    esz = 4 if case["storage"] == "f32" else 2
    vox = case["nx"] * case["ny"] * case["nz"]
    per = 60.0                                   # operations of a sample: position, stencil, table, blend
    cam = _cams(case, 0, 1)[0]
    s = _samples(case, cam)
    px = case["W"] * case["H"] * (16 if case["mode"] == "dvr" else 4)
    seen = min(vox, 8 * s) * esz
    if kind in ("frame", "viewer"):
        return {"bytes": case["views"] * (seen + px), "flops": case["views"] * s * per}
    if kind == "fit":
        v = case["views"]
        g = case.get("voxels", True)
        # voxels copied, bricked and read once; images out, loss gradient in; gradient out
        return {"bytes": vox * 4 * (5 if g else 1) + 3 * v * px, "flops": v * s * per * 3}
    if kind == "ingest":
        return {"bytes": vox * 4 * 2 + vox * 4 + vox * esz + seen + px, "flops": s * per}
    if kind == "compress":
        return {"bytes": vox * 4 * 2 + vox * 4 + 2 * vox * 1.0625 + seen + px, "flops": vox * 14 + s * per}
    b = f = 0.0
    for which, sub, cam, mode, table in _requests(case, 0):
        q = _samples(dict(sub, mode=mode, table=table), cam)
        n = sub["nx"] * sub["ny"] * sub["nz"]
        b += min(n, 8 * q) * (4 if sub["storage"] == "f32" else 2) + cam["W"] * cam["H"] * (16 if mode == "dvr" else 4)
        f += q * per
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------------------------- exact
def _rays(cam, aspect=None):
    """Origins and directions (n, 3), float64 holding the binary32 rays of the pixel centres: which samples
    a ray has is decided in binary32 (one fixed order of operations), everything after it in 64 bits."""
    f = np.float32
    W, H = cam["W"], cam["H"]
    i, j = np.meshgrid(np.arange(W, dtype=f), np.arange(H, dtype=f))
    sx = (i + f(0.5)) / f(W) * f(2) - f(1)
    sy = f(1) - (j + f(0.5)) / f(H) * f(2)
    R, t = cam["view"][:3, :3].astype(f), cam["view"][:3, 3].astype(f)
    asp = f(W) / f(H) if aspect is None else f(aspect)
    z = np.zeros_like(sx)
    if cam["proj"] == 0:
        hh = f(cam["param"]) * f(0.5)
        e = (sx * (hh * asp), sy * hh)
        de = (z, z, z - f(1))
    else:
        th = f(math.tan(float(f(cam["param"])) * 0.5))
        x, y = sx * (th * asp), sy * th
        ln = np.sqrt(x * x + y * y + f(1))
        e, de = (z, z), (x / ln, y / ln, f(-1) / ln)
    y0, y1, y2 = e[0] - t[0], e[1] - t[1], z + (f(0) - t[2])
    o = np.stack([R[0, k] * y0 + R[1, k] * y1 + R[2, k] * y2 for k in range(3)], -1)
    d = np.stack([R[0, k] * de[0] + R[1, k] * de[1] + R[2, k] * de[2] for k in range(3)], -1)
    return o.reshape(-1, 3).astype(np.float64), d.reshape(-1, 3).astype(np.float64)


def _krange(o, d, lo, hi, step):
    """Lattice indices [k0, k1) of each ray inside the box, in binary32."""
    f = np.float32
    o, d, step = o.astype(f), d.astype(f), f(step)
    tin, tout = np.zeros(len(o), f), np.full(len(o), np.inf, f)
    ok = np.ones(len(o), bool)
    with np.errstate(all="ignore"):
        for a in range(3):
            t0, t1 = (f(lo[a]) - o[:, a]) / d[:, a], (f(hi[a]) - o[:, a]) / d[:, a]
            flat = d[:, a] == 0
            ok &= ~flat | ((lo[a] <= o[:, a]) & (o[:, a] < hi[a]))
            tin = np.where(flat, tin, np.maximum(tin, np.minimum(t0, t1)))
            tout = np.where(flat, tout, np.minimum(tout, np.maximum(t0, t1)))
        ok &= (tout > tin) & np.isfinite(tout)
        k0 = np.where(ok, np.ceil(tin / step), 0).astype(np.int64)
        k1 = np.where(ok, np.ceil(tout / step), 0).astype(np.int64)
    return k0, np.maximum(k0, k1)


class _Walk:
    """The samples of all rays of some views, one lattice step of every ray at a time."""

    def __init__(self, cube, case, cams, table, mode):
        self.cube, self.case, self.mode = cube.reshape(-1), case, mode
        self.n = (case["nx"], case["ny"], case["nz"])
        self.win = _window(case) if case["kind"] == "viewer" else ([0, 0, 0], list(self.n))
        self.mask = torch.from_numpy(_mask(case["nz"])).to(DEV) if case["kind"] == "viewer" else None
        self.table = torch.from_numpy(table).to(DEV).double()
        self.dif = torch.cat([self.table[1:] - self.table[:-1], torch.zeros_like(self.table[:1])])
        self.step = float(np.float32(case["step"]))
        rays = [_rays(c) for c in cams]
        o, d = np.concatenate([r[0] for r in rays]), np.concatenate([r[1] for r in rays])
        k0, k1 = _krange(o, d, self.win[0], self.win[1], case["step"])
        self.rays = len(o)
        live = np.nonzero(k1 > k0)[0]
        live = live[np.argsort(k0[live] - k1[live], kind="stable")]      # longest first
        self.live = torch.from_numpy(live).to(DEV)
        self.o, self.d = (torch.from_numpy(v[live]).to(DEV).unbind(1) for v in (o, d))
        self.k0 = torch.from_numpy(k0[live]).to(DEV).double()
        self.count = (k1 - k0)[live]

    def steps(self):
        """(m, sample): the first m rays of the order have a sample at this step."""
        most = int(self.count[0]) if len(self.count) else 0
        ends = np.searchsorted(-self.count, -np.arange(1, most + 1), side="right")
        for j in range(most):
            yield int(ends[j]), j

    def sample(self, m, j):
        """Trilinear value, stencil indices and weights of sample j of the first m rays, and its brick."""
        t = (self.k0[:m] + j) * self.step
        i0, i1, fr, brick = [], [], [], 0
        for a in (2, 1, 0):
            p = self.o[a][:m] + t * self.d[a][:m]
            x = p - 0.5
            fl = torch.floor(x)
            fr.append(x - fl)
            i = fl.long()
            i0.append(i.clamp(0, self.n[a] - 1))
            i1.append((i + 1).clamp(0, self.n[a] - 1))
            brick = brick * 4096 + torch.floor(p / self.case["brick"]).clamp(0, -(-self.n[a] // self.case["brick"]) - 1).long()
        idx, wts = [], []
        for c in range(8):
            q = [i1[k] if (c >> (2 - k)) & 1 else i0[k] for k in range(3)]
            idx.append((q[0] * self.n[1] + q[1]) * self.n[0] + q[2])
            w = [fr[k] if (c >> (2 - k)) & 1 else 1.0 - fr[k] for k in range(3)]
            wts.append(w[0] * w[1] * w[2])
        val = 0
        for c in range(8):
            v = self.cube[idx[c]].double()
            if self.mask is not None:
                z = i1[0] if c >> 2 else i0[0]
                v = torch.where(self.mask[z] != 0, v, torch.full_like(v, float(np.float32(self.case["vmin"]))))
            val = val + wts[c] * v
        return val, idx, wts, brick

    def lookup(self, val):
        lo, hi = float(np.float32(self.case["vmin"])), float(np.float32(self.case["vmax"]))
        n = len(self.table)
        u = (val - lo) / (hi - lo)
        x = u.clamp(0, 1) * (n - 1)
        li = torch.floor(x).long().clamp(0, n - 1)
        lf = x - li
        return self.table[li] + lf[:, None] * self.dif[li], li, lf, (u > 0) & (u < 1)

    def kept(self):
        """Composited samples, step by step: (m, which rays keep it, its value's parts, colour, T before).
        T is the whole ray's; a brick's segment (or with global termination the ray) that has reached the
        threshold takes no more samples."""
        thr = float(np.float32(1.0) - np.float32(min(self.case["tau"], 1.0)))
        k = len(self.live)
        T = torch.ones(k, device=DEV, dtype=torch.float64)
        seg, cur = torch.ones_like(T), torch.full((k,), -1, device=DEV)
        glob = self.case["term"] == "global"
        for m, j in self.steps():
            val, idx, wts, brick = self.sample(m, j)
            if not glob:
                new = brick != cur[:m]
                cur[:m] = brick
                seg[:m] = torch.where(new, torch.ones_like(val), seg[:m])
            on = seg[:m] > thr
            rgba, li, lf, inside = self.lookup(val)
            a = rgba[:, 3] * on
            yield m, on, (val, idx, wts, li, lf, inside), rgba, a, T[:m].clone()
            T[:m] *= 1.0 - a
            seg[:m] *= 1.0 - a
        self.T = T

    def image(self):
        if self.mode == "mip":
            out = torch.full((self.rays,), float(np.float32(self.case["vmin"])), device=DEV, dtype=torch.float64)
            best = torch.full((len(self.live),), -math.inf, device=DEV, dtype=torch.float64)
            for m, j in self.steps():
                best[:m] = torch.maximum(best[:m], self.sample(m, j)[0])
            out[self.live] = best
            return out
        acc = torch.zeros((len(self.live), 3), device=DEV, dtype=torch.float64)
        self.T = torch.ones(len(self.live), device=DEV, dtype=torch.float64)
        for m, on, _, rgba, a, T in self.kept():
            acc[:m] += (T * a)[:, None] * rgba[:, :3]
        out = torch.zeros((self.rays, 4), device=DEV, dtype=torch.float64)
        out[self.live] = torch.cat([acc, 1.0 - self.T[:, None]], 1)
        return out

    def gradient(self, img, gout, voxels):
        """d/d(table), d/d(voxels) of sum(img * gout) with the stops held fixed."""
        g, fin = gout[self.live], img[self.live]
        gt = torch.zeros((512 * len(self.table), 4), device=DEV, dtype=torch.float64)
        gv = torch.zeros(self.cube.numel(), device=DEV, dtype=torch.float64) if voxels else None
        n = len(self.table)
        lane = torch.arange(len(self.live), device=DEV) % 512 * n
        acc = torch.zeros((len(self.live), 3), device=DEV, dtype=torch.float64)
        scale = (n - 1) / (float(np.float32(self.case["vmax"])) - float(np.float32(self.case["vmin"])))
        for m, on, (val, idx, wts, li, lf, inside), rgba, a, T in self.kept():
            w = (T * a)[:, None]
            acc[:m] += w * rgba[:, :3]
            gm = g[:m]
            rest = (gm[:, :3] * (fin[:m, :3] - acc[:m])).sum(1)
            ga = T * (gm[:, :3] * rgba[:, :3]).sum(1) + (gm[:, 3] * (1.0 - fin[:m, 3]) - rest) / (1.0 - a)
            gs = torch.cat([w * gm[:, :3], ga[:, None]], 1) * on[:, None]
            gt.index_add_(0, lane[:m] + li, gs * (1.0 - lf)[:, None])
            gt.index_add_(0, lane[:m] + (li + 1).clamp(max=n - 1), gs * lf[:, None])
            if voxels:
                dv = (gs * self.dif[li]).sum(1) * scale * inside
                for c in range(8):
                    gv.index_add_(0, idx[c], dv * wts[c])
        return gt.view(512, n, 4).sum(0), gv


def _pictures(cube, case, cams, table="ramp", mode="dvr"):
    out = []
    for cam in cams:
        w = _Walk(cube, dict(case, W=cam["W"], H=cam["H"]), [cam], _table(table), mode)
        im = w.image()
        out.append(im.view(cam["H"], cam["W"], 4) if mode == "dvr" else im.view(cam["H"], cam["W"]))
    return out


def _wavelet(cube):
    """The cube after a round trip through 8^3 Haar blocks with int8 details (power-of-two step per
    subband, block averages kept)."""
    nz, ny, nx = cube.shape
    out = torch.empty_like(cube, dtype=torch.float64)
    yy, xx = (torch.arange(-(-m // 8) * 8, device=DEV).clamp(max=m - 1) for m in (ny, nx))
    for z0 in range(0, nz, 32):
        zz = torch.arange(z0, min(z0 + 32, -(-nz // 8) * 8), device=DEV).clamp(max=nz - 1)
        b = cube[zz][:, yy][:, :, xx].double()
        shp = b.shape
        b = b.view(shp[0] // 8, 8, shp[1] // 8, 8, shp[2] // 8, 8).permute(0, 2, 4, 1, 3, 5).reshape(-1, 8, 8, 8)
        levels = []
        for _ in range(3):
            bands = [b]
            for ax in (3, 2, 1):
                ev, od = (slice(0, None, 2), slice(1, None, 2))
                pick = lambda v, s: v[(slice(None),) * ax + (s,)]   # noqa: E731
                bands = [h for v in bands for h in ((pick(v, ev) + pick(v, od)) / 2, (pick(v, ev) - pick(v, od)) / 2)]
            q = [bands[0]]
            for v in bands[1:]:
                m = v.abs().amax((1, 2, 3), keepdim=True)
                e = torch.ceil(torch.log2(m.clamp(min=1e-300) / 127.0)).clamp(-126, 120)
                st = torch.exp2(e)
                q.append(torch.where(m > 0, torch.round(v / st).clamp(-127, 127) * st, torch.zeros_like(v)))
            levels.append(q)
            b = bands[0]
        for q in reversed(levels):
            bands = [b] + q[1:]
            for ax in (1, 2, 3):
                nxt = []
                for s, d in zip(bands[::2], bands[1::2]):
                    sh = list(s.shape)
                    sh[ax] *= 2
                    nxt.append(torch.stack([s + d, s - d], ax + 1).reshape(sh))
                bands = nxt
            b = bands[0]
        b = b.view(shp[0] // 8, shp[1] // 8, shp[2] // 8, 8, 8, 8).permute(0, 3, 1, 4, 2, 5).reshape(shp)
        h = min(32, nz - z0)
        out[z0:z0 + h] = b[:h, :ny, :nx]
    return out


def exact(case, seed):
    kind = case["kind"]
    cube = _case_cube(case, seed)
    if kind == "frame":
        return [v.cpu() for v in _pictures(cube, case, _cams(case, seed, case["views"]), case["table"], case["mode"])]
    if kind == "viewer":
        return _pictures(cube, case, _cams(case, seed, 1), case["table"])[0].cpu()
    if kind == "ingest":
        img = _pictures(cube, case, _cams(case, seed, 1), case["table"])[0]
        return {"range": np.array([float(cube.min()), float(cube.max())]), "img": img.cpu()}
    if kind == "compress":
        return _pictures(_wavelet(cube), case, _cams(case, seed, 1), case["table"])[0].cpu()
    if kind == "fit":
        w = _Walk(cube, case, _cams(case, seed, case["views"]), _table(case["table"]), "dvr")
        img = w.image()
        shape = (case["views"], case["H"], case["W"], 4)
        vox = case.get("voxels", True)
        gt, gv = w.gradient(img, img - _targets(case, seed).double().view(-1, 4), vox)
        return {"img": img.view(shape).cpu(), "table": gt.cpu(),
                "voxels": gv.view(case["nz"], case["ny"], case["nx"]).cpu() if vox else None}
    sub = _second(case)
    cubes = [cube, _cube(sub["nx"], sub["ny"], sub["nz"], case["data"], case["noise"], seed + 3)]
    return [_pictures(cubes[which], dict(s, kind="frame"), [cam], table, mode)[0].cpu()
            for which, s, cam, mode, table in _requests(case, seed)]
