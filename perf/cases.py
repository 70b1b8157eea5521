"""What is measured: the calls a program makes, over the range of sizes it makes them at.

A case is one of

  frame    one frame of a running session (`dof.frame`): the whole depth-of-field pass, with its
           history in a steady state and the camera on its way (or still, for the small preview)
  batch    one step of several sessions together (`dof.batch_frame`), or the same step replayed as
           a captured graph (`dof.Graph`)
  gbuffer  the ray-cast G-buffer producer (`dof.gbuffer`)
  raster   the object-order G-buffer producer (`dof.gbuffer_raster`)
  upload   new geometry: the scene upload with its tree build (`dof.Scene`) and the first G-buffer
           from it
  tiles    the allocation-free tile map (`dof.coc_tiles_noalloc`)

Scenes, lenses and parameters are the repository's own workloads (`synth`), at other seeds.
`settings`: "default" is a context as it is created; "tuned" pins what the autotuners pick for the
workloads (warp packets over the binary tree, the gathers' shapes), as a session that has been
tuned at its start runs.
"""

import math

import numpy as np
import torch

from paper_2210_06158_gb300 import dof
from synth import make_workload
from synth.scenes import Camera, scene_grass_field, taa_jitter

DEVICE = "cuda:0"

# what the tuners leave on a context, by lens (pixel order at 1 spp and in the adaptive mode,
# lens cells of 1/8 aperture at several rays per pixel)
TUNED = {
    "c1": dict(ploc=96, trace=dict(packets=1, bvh_width=2, ray_grid=1, stack=32, stats=0),
               gather=dict(block=(32, 8), main_form=0, recon_block=(32, 8))),
    "c2": dict(ploc=96, trace=dict(packets=1, bvh_width=2, ray_grid=1, stack=32, stats=0),
               gather=dict(block=(64, 4), main_form=3, recon_block=(32, 8))),
    "c3": dict(ploc=48, trace=dict(packets=1, bvh_width=2, ray_grid=8, stack=32, stats=0),
               gather=dict(block=(32, 4), main_form=1, recon_block=(16, 16))),
}


def _frame(name, lens, width, height, **over):
    c = dict(name=name, kind="frame", lens=lens, width=width, height=height, tris=0, spp=1, m=0, storage=0,
             half_gbuffer=False, blades=0, taa=False, settings="default")
    c.update(over)
    if name is None:
        del c["name"]
    return c


def listed():
    return [
        # an engine asks for the tile map of its depth buffer each frame, without any allocation
        dict(name="tile_map_4k", kind="tiles", lens="c3", width=3840, height=2160),
        # a small preview, still camera: launches and latency
        _frame("frame_144p", "c1", 256, 144),
        # an odd window size with a hexagonal diaphragm and the adaptive ray budget, light scene
        _frame("frame_768p_adaptive_hex", "c2", 1366, 768, tris=100_000, m=4, blades=6),
        # the 1080p workload as a first-time user runs it
        _frame("frame_1080p", "c2", 1920, 1080, tris=500_000),
        # the same in a tuned session with half-precision images
        _frame("frame_1080p_half_tuned", "c2", 1920, 1080, tris=500_000, storage=1, half_gbuffer=True, settings="tuned"),
        # the adaptive ray budget of up to ten rays per pixel, tuned
        _frame("frame_1080p_adaptive_tuned", "c2", 1920, 1080, tris=500_000, m=10, settings="tuned"),
        # a jittered camera with the final anti-aliasing pass
        _frame("frame_1440p_taa", "c2", 2560, 1440, tris=300_000, taa=True),
        # the 4K workload, four rays per pixel through a wide lens, tuned
        _frame("frame_2160p_tuned", "c3", 3840, 2160, tris=2_000_000, spp=4, settings="tuned"),
        # a server's step: eight sessions of four sizes
        dict(name="batch_8_sessions", kind="batch", graph=False, sessions=8, width=1280, height=720, tris=200_000,
             settings="default"),
        # the renderer's G-buffer, by rays and by triangles
        dict(name="gbuffer_1080p", kind="gbuffer", lens="c2", width=1920, height=1080, tris=500_000),
        dict(name="raster_1080p", kind="raster", lens="c2", width=1920, height=1080, tris=500_000),
        # geometry that changes: upload, tree build, first view
        dict(name="upload_500k", kind="upload", lens="c2", width=640, height=360, tris=500_000),
    ]


def _size(rng, lo, hi):
    """An even size of between lo and hi lines, spread over the logarithm, of some aspect ratio."""
    h = int(math.exp(rng.uniform(math.log(lo), math.log(hi)))) // 2 * 2
    w = int(h * rng.choice((4 / 3, 1.6, 16 / 9, 21 / 9 if h <= 1600 else 16 / 9))) // 2 * 2
    return w, h


def draw(rng):
    kind = rng.choice(("frame",) * 6 + ("batch", "gbuffer", "raster", "upload", "tiles"))
    tris = int(math.exp(rng.uniform(math.log(30_000), math.log(500_000))))
    if kind == "frame":
        lens = rng.choice(("c1", "c2", "c2", "c3"))
        w, h = _size(rng, 144, 720 if lens == "c1" else 2160)
        adaptive = rng.random() < 0.3
        return _frame(None, lens, w, h, tris=0 if lens == "c1" else tris * (2 if lens == "c3" else 1),
                      spp=1 if adaptive else rng.choice((1, 1, 2, 4)), m=rng.randint(2, 10) if adaptive and h <= 1080 else 0,
                      storage=rng.choice((0, 0, 1)), half_gbuffer=rng.random() < 0.3,
                      blades=rng.choice((0, 0, 0, 3, 5, 6, 8)), taa=rng.random() < 0.25,
                      settings=rng.choice(("default", "tuned")))
    if kind == "batch":
        w, h = _size(rng, 180, 720)
        return dict(kind=kind, graph=rng.random() < 0.5, sessions=rng.randint(2, 8), width=w, height=h, tris=min(tris, 200_000),
                    settings=rng.choice(("default", "tuned")))
    if kind == "tiles":
        w, h = _size(rng, 180, 2160)
        return dict(kind=kind, lens=rng.choice(("c2", "c3")), width=w, height=h)
    w, h = _size(rng, 180, 360 if kind == "upload" else 1080)
    return dict(kind=kind, lens=rng.choice(("c1", "c2", "c3")), width=w, height=h, tris=tris)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _workload(lens, width, height, tris, seed, frames):
    """The workload `lens` at another size, triangle count and seed, with `frames` poses."""
    w = make_workload(lens, W=width, H=height, n_frames=None if lens == "c1" else frames, session=seed)
    if lens != "c1" and tris:
        f_m, near = w.intr["f_m"], (1.2, 4.7) if lens == "c2" else (1.3, 4.8)
        scene_seed = w.params["albedo_seed"]
        w.scene_fn = lambda: scene_grass_field(scene_seed, tris / 500_000, f_m=f_m, near=near)
    return w


def _cameras(w, jittered):
    """The cameras of one turn along the workload's path and back, each after the one before it."""
    n = w.n_frames
    path = list(range(n)) + list(range(n - 2, 0, -1))
    cams = []
    for k, at in enumerate(path):
        prev = path[k - 1]
        cam = Camera.from_poses(w.intr, w.poses[at], w.poses[prev], frame_index=k)
        if jittered:
            cam.jitter, cam.prev_jitter = taa_jitter(k), taa_jitter((k - 1) % len(path))
        cams.append(cam)
    return cams


def _context(settings, lens):
    ctx = dof.Context(0)
    if settings == "tuned":
        t = TUNED[lens]
        ctx.set_ploc_radius(t["ploc"])
        ctx.set_trace(**t["trace"])
        ctx.set_gather(**t["gather"])
    return ctx


class _Plane:
    """A history's device buffer as a tensor (the history lives as long as the tensor does)."""

    def __init__(self, hist, name, shape):
        ptr, n = hist.buffer(name)
        assert n == 4 * int(np.prod(shape))
        self.hist = hist
        self.__cuda_array_interface__ = dict(shape=tuple(shape), typestr="<f4", data=(ptr, False), version=3)


def _state_planes(hist):
    n = (hist.width // 2) * (hist.height // 2)
    return (torch.as_tensor(_Plane(hist, "HIST", (3, n, 4)), device=DEVICE),
            torch.as_tensor(_Plane(hist, "VAR_BLUR", (n,)), device=DEVICE))


WARM = 3        # frames a session has run before its pass is measured


class _Session:
    """One viewer: scene, cameras, their G-buffers and the running history."""

    def __init__(self, ctx, w, params, half_gbuffer=False, jittered=False):
        self.ctx, self.params, self.k = ctx, params, 0
        self.scene = dof.Scene(ctx, w.scene)
        self.cams = _cameras(w, jittered)
        self.gbufs = []
        for cam in self.cams:
            g = dof.gbuffer(ctx, self.scene, cam, params, w.W, w.H)
            del g["prim"]
            if params["ray_mode"] == 0:
                del g["normal"]
            if half_gbuffer:
                for p in ("color", "normal"):
                    if p in g:
                        g[p] = g[p].half()
            self.gbufs.append(g)
        self.structs = [dof.camera_struct(c) for c in self.cams]
        self.params_s = dof.params_struct(params)
        rays = params["m"] if params["ray_mode"] else params["spp"]
        self.hist = dof.History(ctx, w.W, w.H, max_rays=rays, taa=params["taa_alpha"] > 0)
        self.out = torch.empty((w.H, w.W, 4), dtype=torch.float32, device=DEVICE)

    def next(self):
        """The next frame's G-buffer and camera."""
        at = self.k % len(self.cams)
        cam = self.structs[at]
        cam.frame_index = self.k
        self.k += 1
        return self.gbufs[at], cam

    def frame(self):
        g, cam = self.next()
        return dof.frame(self.ctx, self.scene, g, None, None, self.hist, out=self.out, cam_struct=cam,
                         params_s=self.params_s)

    def item(self):
        g, cam = self.next()
        return dict(scene=self.scene, gbuf=g, cam=cam, params=self.params_s, hist=self.hist, out=self.out)

    def settle(self, step):
        """Runs the warm-up frames; keeps the two history buffers that frames write in turn."""
        self.planes = [None, None]
        for _ in range(WARM):
            step()
            self.planes[self.k & 1] = _state_planes(self.hist)


def _params(w, case):
    over = dict(image_storage=case.get("storage", 0), aperture_blades=case.get("blades", 0), spp=case.get("spp", 1))
    if case.get("m"):
        over.update(ray_mode=1, m=case["m"])
    if case.get("taa"):
        over.update(taa_alpha=0.1)
    return dict(w.params, **over)


def prepare(case, seed):
    kind = case["kind"]
    seed = int(seed)
    if kind == "frame":
        w = _workload(case["lens"], case["width"], case["height"], case["tris"], seed, 4)
        s = _Session(_context(case["settings"], case["lens"]), w, _params(w, case), case["half_gbuffer"], case["taa"])
        s.settle(s.frame)
        return dict(case=case, session=s)
    if kind == "batch":
        # sizes in thirds from the given one up to twice it, scenes from the given count down to a half
        ctx = _context(case["settings"], "c2")
        ss = []
        for i in range(case["sessions"]):
            f = (3 + i % 4) / 3
            w = _workload("c2", int(case["width"] * f) // 2 * 2, int(case["height"] * f) // 2 * 2,
                          case["tris"] // (1 + i % 2), seed * 64 + i, 2)
            ss.append(_Session(ctx, w, _params(w, case)))
        state = dict(case=case, ctx=ctx, sessions=ss, graph=None)
        for s in ss:
            s.settle(s.frame)
        if case["graph"]:
            state["graph"] = dof.Graph(ctx, [s.item() for s in ss])
            for s in ss:
                s.k -= 1        # the capture ran nothing
        return state
    if kind == "tiles":
        w = _workload("c1", case["width"], case["height"], 0, seed, 1)
        lens = make_workload(case["lens"], n_frames=1)
        ctx = dof.Context(0)
        depth = dof.gbuffer(ctx, dof.Scene(ctx, w.scene), w.camera(0), w.params, w.W, w.H)["depth"]
        cam = lens.camera(0)
        cam.focus_m = cam.focus_m * (0.5 + (seed % 97) / 97)
        # the first call in a context loads the device code (a session's start)
        dof.coc_tiles_noalloc(depth, cam, lens.params)
        tw, th = -(-(w.W // 2) // 8), -(-(w.H // 2) // 8)
        return dict(case=case, ctx=ctx, depth=depth, cam=cam, params=lens.params,
                    out=torch.empty((th, tw, 2), dtype=torch.float32, device=DEVICE))
    w = _workload(case["lens"], case["width"], case["height"], case["tris"], seed, 4)
    ctx = dof.Context(0)
    cams = [Camera.from_poses(w.intr, p) for p in w.poses]
    state = dict(case=case, ctx=ctx, host=w.scene, cams=cams, params=w.params, k=0)
    if kind != "upload":
        state["scene"] = dof.Scene(ctx, w.scene)
        P = (w.H, w.W)
        state["out"] = dict(color=torch.empty(P + (4,), device=DEVICE), depth=torch.empty(P, device=DEVICE),
                            normal=torch.empty(P + (4,), device=DEVICE),
                            prim=torch.empty(P, dtype=torch.int32, device=DEVICE))
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "frame":
        s = state["session"]
        out = s.frame()
        hist, var = s.planes[s.k & 1]
        return dict(image=out, history=hist, variance=var)
    if kind == "batch":
        items = [s.item() for s in state["sessions"]]
        outs = state["graph"].launch(items) if state["graph"] else dof.batch_frame(state["ctx"], items)
        planes = [s.planes[s.k & 1] for s in state["sessions"]]
        return dict(images=outs, histories=[p[0] for p in planes], variances=[p[1] for p in planes])
    if kind == "tiles":
        return dof.coc_tiles_noalloc(state["depth"], state["cam"], state["params"], out=state["out"])
    cam = state["cams"][state["k"] % len(state["cams"])]
    state["k"] += 1
    if kind == "upload":
        state["scene"] = dof.Scene(state["ctx"], state["host"])
        return dof.gbuffer(state["ctx"], state["scene"], cam, state["params"], case["width"], case["height"])
    return dof.gbuffer(state["ctx"], state["scene"], cam, state["params"], case["width"], case["height"], out=state["out"],
                       raster=kind == "raster")


# ---------------------------------------------------------------------------
# the work a pass cannot do without
# ---------------------------------------------------------------------------

def _frame_work(width, height, rays_per_px, normals, half, taa):
    P, N = width * height, width * height // 4
    # colour and depth (and normals) read, the image written; the history (12 floats) and the
    # blurred variance read and written per half-resolution pixel; the previous image with TAA
    byte = P * (8 if half else 16) + 4 * P + (P * (8 if half else 16) if normals else 0) + 16 * P + 2 * 52 * N + (32 * P if taa else 0)
    # the two 81-tap gathers (a bilinear tap of five values and its weights; a trilinear tap of
    # six), and a descent of ~20 levels with two boxes each and a few triangles per ray
    flop = N * 81 * (82 + 134) + N * rays_per_px * (20 * 47 + 4 * 48)
    return byte, flop


def work(case):
    kind = case["kind"]
    P = case["width"] * case["height"]
    if kind == "frame":
        b, f = _frame_work(case["width"], case["height"], case["m"] / 2 or case["spp"], case["m"] > 0, case["half_gbuffer"],
                           case["taa"])
    elif kind == "batch":
        b = f = 0
        for i in range(case["sessions"]):
            s = (3 + i % 4) / 3
            x, y = _frame_work(int(case["width"] * s), int(case["height"] * s), 1, False, False, False)
            b, f = b + x, f + y
    elif kind == "tiles":
        b, f = 4 * P + 8 * P / 256, 8 * P / 4
    else:
        tris = case["tris"] if case["lens"] != "c1" else 2802
        b, f = 40 * P, P * (20 * 47 + 4 * 48)
        if kind == "raster":
            b += 48 * tris
        if kind == "upload":
            # vertices, indices and materials in; triangles, nodes and the index out
            b += tris * (1.6 * 12 + 12 + 4) + tris * (48 + 64 + 64 + 4)
            f += tris * 200
    return dict(bytes=b, flops=f)


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------
# The tile map, and G-buffers and still-camera frames of the small scene, in plain torch float64.
# The other cases trace hundreds of thousands of triangles: None.

F64 = torch.float64


def _t(x):
    return torch.as_tensor(np.asarray(x, dtype=np.float64), dtype=F64, device=DEVICE)


def _coc(cam, width, z):
    f, n, d, ws = (float(np.float32(v)) for v in (cam.f_m, cam.f_number, cam.focus_m, cam.sensor_w_m))
    return f / n * f * width / (ws * (d - f)) * (z - d) / z


def _half_depth(depth, cam, params):
    """Nearest depth of each 2x2 block, and its clamped signed CoC radius (half-resolution px)."""
    H, W = depth.shape
    z = depth.to(F64).clamp(max=params["z_far_m"]).view(H // 2, 2, W // 2, 2).amin((1, 3))
    r = params["max_coc_px"] / 2
    return z, (_coc(cam, W, z) / 4).clamp(-r, r)


def _dilated(rho, params):
    """Maxima of (near radius, |radius|) over 8x8 tiles, dilated over the reach of the largest one."""
    v = torch.stack(((-rho).clamp(min=0), rho.abs()))[None]
    h, w = rho.shape
    v = torch.nn.functional.pad(v, (0, -w % 8, 0, -h % 8))
    v = torch.nn.functional.max_pool2d(v, 8)
    k = math.ceil(params["max_coc_px"] / 2 / 8)
    return torch.nn.functional.max_pool2d(v, 2 * k + 1, stride=1, padding=k)[0].permute(1, 2, 0)


def _dirs(cam, width, height, x, y):
    """Unit directions through sensor points (x, y) and the lens centre."""
    f, d, ws = (float(np.float32(v)) for v in (cam.f_m, cam.focus_m, cam.sensor_w_m))
    F = width * (f * d / (d - f)) / ws
    sx, sy = (x - width / 2) / F, (y - height / 2) / F
    v = _t(cam.fwd) + sx[..., None] * _t(cam.right) - sy[..., None] * _t(cam.up)
    return v / v.norm(dim=-1, keepdim=True)


def _closest(scene, O, D):
    """Closest hits (t, triangle or -1) of rays from O along D: every ray against every triangle."""
    v = _t(scene.verts)[torch.as_tensor(scene.tris.astype(np.int64), device=DEVICE)]
    e1, e2 = v[:, 1] - v[:, 0], v[:, 2] - v[:, 0]
    best_t, best_k = [], []
    for o, d in zip(O.split(4096), D.split(4096)):
        p = torch.linalg.cross(d[:, None], e2[None])
        det = (p * e1).sum(-1)
        s = o[:, None] - v[None, :, 0]
        u = (s * p).sum(-1) / det
        q = torch.linalg.cross(s, e1[None].expand_as(s))
        w = (q * d[:, None]).sum(-1) / det
        t = (q * e2).sum(-1) / det
        t = torch.where((det != 0) & (u >= 0) & (w >= 0) & (u + w <= 1) & (t > 0), t, math.inf)
        m, k = t.min(1)
        best_t.append(m)
        best_k.append(torch.where(m.isinf(), -1, k))
    return torch.cat(best_t), torch.cat(best_k)


def _fmix(h):
    h = np.asarray(h, dtype=np.uint32)
    h = (h ^ (h >> np.uint32(16))) * np.uint32(0x85EBCA6B)
    h = (h ^ (h >> np.uint32(13))) * np.uint32(0xC2B2AE35)
    return h ^ (h >> np.uint32(16))


def _shade(scene, params, k, D):
    """Colour and outward normal of hits on triangles k (-1: sky, zero normal)."""
    n_tri = scene.n_tris
    with np.errstate(over="ignore"):
        base = _fmix(np.uint32(int(params["albedo_seed"]) & 0xFFFFFFFF))
        albedo = 0.1 + 0.8 * (_fmix(base ^ np.arange(3 * n_tri, dtype=np.uint32)) >> np.uint32(8)).astype(np.float64) / 2 ** 24
    albedo = _t(albedo.reshape(n_tri, 3))
    v = _t(scene.verts)[torch.as_tensor(scene.tris.astype(np.int64), device=DEVICE)]
    n = torch.linalg.cross(v[:, 1] - v[:, 0], v[:, 2] - v[:, 0])
    n = n / n.norm(dim=-1, keepdim=True)
    hit = k >= 0
    kk = k.clamp(min=0)
    n = n[kk]
    n = torch.where((n * D).sum(-1, keepdim=True) > 0, -n, n)
    light = _t(params["light_dir"])
    lam = (-(n * (light / light.norm()))).sum(-1).clamp(min=0)
    col = albedo[kk] * (params["k_a"] + params["k_d"] * lam)[:, None]
    emits = torch.as_tensor(scene.mat.astype(np.int64), device=DEVICE)[kk] == 1
    col = torch.where(emits[:, None], params["emit"] * albedo[kk], col)
    return torch.where(hit[:, None], col, _t(params["sky"])), torch.where(hit[:, None], n, 0.0)


def _exact_gbuffer(w, cam):
    y, x = torch.meshgrid(torch.arange(w.H, device=DEVICE), torch.arange(w.W, device=DEVICE), indexing="ij")
    D = _dirs(cam, w.W, w.H, x.to(F64) + 0.5, y.to(F64) + 0.5).reshape(-1, 3)
    t, k = _closest(w.scene, _t(cam.pos).expand_as(D), D)
    col, n = _shade(w.scene, w.params, k, D)
    one = torch.ones_like(t)[:, None]
    depth = t * (D * _t(cam.fwd)).sum(-1)
    return dict(color=torch.cat((col, one), 1).view(w.H, w.W, 4), depth=depth.view(w.H, w.W),
                normal=torch.cat((n, 0 * one), 1).view(w.H, w.W, 4), prim=None)


def _lens_samples(n, spp, frame, params):
    """The two uniforms of each (pixel, sample): Philox4x64-10 in numpy."""
    u64 = np.uint64

    def mulhilo(a, b):
        lo32 = u64(0xFFFFFFFF)
        a0, a1, b0, b1 = a & lo32, a >> u64(32), b & lo32, b >> u64(32)
        m0, m1, m2 = a0 * b0, a1 * b0, a0 * b1
        mid = (m0 >> u64(32)) + (m1 & lo32) + (m2 & lo32)
        return a1 * b1 + (m1 >> u64(32)) + (m2 >> u64(32)) + (mid >> u64(32)), a * b

    with np.errstate(over="ignore"):
        q, s = np.meshgrid(np.arange(n, dtype=np.uint64), np.arange(spp, dtype=np.uint64), indexing="ij")
        c = [q, s, np.full_like(q, frame), np.zeros_like(q)]
        key = [int(params["seed"]) & (2 ** 64 - 1), int(params["session"]) & (2 ** 64 - 1)]
        for r in range(10):
            k0 = u64((key[0] + r * 0x9E3779B97F4A7C15) % 2 ** 64)
            k1 = u64((key[1] + r * 0xBB67AE8584CAA73B) % 2 ** 64)
            h0, l0 = mulhilo(u64(0xD2E7470EE14C6C93), c[0])
            h1, l1 = mulhilo(u64(0xCA5A826395121157), c[2])
            c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
    return tuple(_t((x >> u64(40)).astype(np.float64) / 2 ** 24) for x in c[:2])


def _bilinear(img, x, y):
    """img (H, W, C) at (x, y), texel centres at integers, clamped to the edge."""
    h, w = img.shape[:2]
    xf, yf = x.floor(), y.floor()
    fx, fy = (x - xf)[..., None], (y - yf)[..., None]
    xa, xb = xf.long().clamp(0, w - 1), (xf.long() + 1).clamp(0, w - 1)
    ya, yb = yf.long().clamp(0, h - 1), (yf.long() + 1).clamp(0, h - 1)
    return (img[ya, xa] * (1 - fx) + img[ya, xb] * fx) * (1 - fy) + (img[yb, xa] * (1 - fx) + img[yb, xb] * fx) * fy


def _rings():
    yield 0.0, 0.0, 0.0
    for k in range(1, 5):
        for m in range(8 * k):
            a = 2 * math.pi * m / (8 * k)
            yield math.cos(a), math.sin(a), k / 4


def _neighbours(img, reach):
    """The (2 reach + 1)^2 clamped neighbourhoods of img (H, W, C), stacked first, and which lie inside."""
    h, w = img.shape[:2]
    y, x = torch.meshgrid(torch.arange(h, device=DEVICE), torch.arange(w, device=DEVICE), indexing="ij")
    v, inside = [], []
    for dy in range(-reach, reach + 1):
        for dx in range(-reach, reach + 1):
            yy, xx = y + dy, x + dx
            inside.append((yy >= 0) & (yy < h) & (xx >= 0) & (xx < w))
            v.append(img[yy.clamp(0, h - 1), xx.clamp(0, w - 1)])
    return torch.stack(v), torch.stack(inside)


def _exact_frame(w, cam, params, color, depth, frame, hist):
    """One frame with a still camera: (image, new history planes, blurred variance)."""
    H, W = depth.shape
    h, wd = H // 2, W // 2
    sat = lambda v: v.clamp(0, 1)  # noqa: E731
    lum = _t((0.2126, 0.7152, 0.0722))
    gy, gx = torch.meshgrid(torch.arange(h, device=DEVICE, dtype=F64), torch.arange(wd, device=DEVICE, dtype=F64), indexing="ij")
    rmax, cover = params["max_coc_px"] / 2, 1 / params["cover_ramp_px"]
    # post-process: downscale, tiles, prefilter, main filter, median
    z, rho = _half_depth(depth, cam, params)
    rgb = color[..., :3].to(F64).view(h, 2, wd, 2, 3).mean((1, 3))
    tiles = _dilated(rho, params)
    tile = tiles.repeat_interleave(8, 0).repeat_interleave(8, 1)[:h, :wd]
    near, R = tile[..., 0], tile[..., 1]
    img = torch.cat((rgb, rho[..., None]), -1)
    acc, ws = rgb.clone(), torch.ones_like(z)
    rp = (R / 8).clamp(min=math.sqrt(0.5))
    for k in range(8):
        s = _bilinear(img, gx + rp * math.cos(k * math.pi / 4), gy + rp * math.sin(k * math.pi / 4))
        wt = sat(1 - (s[..., 3] - rho).abs() / rho.abs().clamp(min=1))
        acc, ws = acc + wt[..., None] * s[..., :3], ws + wt
    pre = torch.cat((acc / ws[..., None], rho[..., None], z[..., None]), -1)
    acc, ws = torch.zeros((h, wd, 4), dtype=F64, device=DEVICE), torch.zeros_like(z)
    for ux, uy, ur in _rings():
        s = _bilinear(pre, gx + ur * R * ux, gy + ur * R * uy)
        ri, dist = s[..., 3].abs(), ur * R
        wf = sat((z - s[..., 4]) / params["depth_range_m"])
        a = 1 / (math.pi * ri.clamp(min=math.pi ** -0.5) ** 2)
        wt = (wf * sat((ri - dist) * cover + 0.5) + (1 - wf) * sat((torch.minimum(ri, rho.abs()) - dist) * cover + 0.5)) * a
        bright = sat(((s[..., :3] * lum).sum(-1) - params["bright_lum"]) / params["bright_ramp"])
        acc, ws = acc + wt[..., None] * torch.cat((s[..., :3], bright[..., None]), -1), ws + wt
    pp = _neighbours(acc / ws[..., None], 1)[0].median(0).values
    # rays: lens samples, closest hits, shading, the near/far split
    mask = near >= params["mask_near_hpx"]
    n, spp = h * wd, params["spp"]
    u1, u2 = _lens_samples(n, spp, frame, params)
    O, Rt, Up, Fw = _t(cam.pos), _t(cam.right), _t(cam.up), _t(cam.fwd)
    dp = _dirs(cam, W, H, 2 * gx + 1, 2 * gy + 1).reshape(-1, 1, 3)
    focus = O + (float(np.float32(cam.focus_m)) / (dp * Fw).sum(-1, keepdim=True)) * dp
    r = u1.sqrt()[..., None] * (float(np.float32(cam.f_m)) / float(np.float32(cam.f_number)) / 2)
    L = O + r * torch.cos(2 * math.pi * u2)[..., None] * Rt + r * torch.sin(2 * math.pi * u2)[..., None] * Up
    D = focus - L
    D = (D / D.norm(dim=-1, keepdim=True)).reshape(-1, 3)
    L = L.reshape(-1, 3)
    t, k = _closest(w.scene, L, D)
    col, _ = _shade(w.scene, params, k, D)
    hit, along = k >= 0, (D * Fw).sum(-1)
    zr = torch.where(hit, (t * along).clamp(max=params["z_far_m"]), params["z_far_m"])
    c = _coc(cam, W, zr)
    rad = (c / 4).clamp(-rmax, rmax).abs()
    wn = sat(-c / math.sqrt(2))
    mean = lambda v: v.view(h, wd, spp, -1).mean(2)  # noqa: E731
    cur = torch.cat((mean(wn[:, None] * col), mean(wn), mean((1 - wn)[:, None] * col), 1 - mean(wn), mean(wn * rad),
                     mean((1 - wn) * rad)), -1)
    # accumulation: the still camera keeps every pixel in place
    L_cur = ((cur[..., 0:3] + cur[..., 4:7]) * lum).sum(-1)
    if hist is None:
        W_h, old = torch.zeros_like(z), torch.zeros((h, wd, 12), dtype=F64, device=DEVICE)
    else:
        old = hist
        W_h = (old[..., 3] + old[..., 7] > 0).to(F64)
    a = params["alpha"] * W_h
    ema = a[..., None] * old[..., :10] + (1 - a)[..., None] * cur
    mu = a * old[..., 10] + (1 - a) * L_cur
    var = (1 - a) * (L_cur - mu) ** 2 + a * (old[..., 11] + (old[..., 10] - mu) ** 2)
    new = torch.where(mask[..., None], torch.cat((ema, mu[..., None], var[..., None]), -1), 0.0)
    tot = (new[..., 3] + new[..., 7]).clamp(min=1e-300)
    crt = torch.where(mask[..., None], torch.cat((new[..., 0:3] + new[..., 4:7], new[..., 3:4]), -1) / tot[..., None], 0.0)
    ct = torch.where(mask, (new[..., 8] + new[..., 9]) / tot, 0.0)
    b5 = _t((1, 4, 6, 4, 1))
    nb, _ = _neighbours(new[..., 11:12], 2)
    var_blur = (nb[..., 0] * (b5[:, None] * b5[None]).reshape(25, 1, 1)).sum(0) / 256
    # lower median over the neighbours with rays
    nb, inside = _neighbours(torch.cat((crt, mask[..., None].to(F64)), -1), 1)
    ok = inside & (nb[..., 4] > 0)
    srt = torch.where(ok[..., None], nb[..., :3], math.inf).sort(0).values
    at = ((ok.sum(0) - 1).clamp(min=0) // 2)[None, ..., None].expand(1, h, wd, 3)
    med = torch.where(mask[..., None], torch.cat((srt.gather(0, at)[0], crt[..., 3:4]), -1), 0.0)
    # the pyramid and the reconstruction
    v = mask[..., None].to(F64)
    mips = [torch.cat((med * v, ct[..., None] * v, v), -1)]
    levels = max(1, min(4, math.ceil(params["lod_max"]) + 1))
    for _ in range(levels - 1):
        m = mips[-1]
        mh, mw = m.shape[:2]
        yy = (2 * torch.arange((mh + 1) // 2, device=DEVICE)[:, None] + torch.tensor((0, 1), device=DEVICE)).clamp(max=mh - 1)
        xx = (2 * torch.arange((mw + 1) // 2, device=DEVICE)[:, None] + torch.tensor((0, 1), device=DEVICE)).clamp(max=mw - 1)
        mips.append(sum(m[yy[:, i]][:, xx[:, j]] for i in (0, 1) for j in (0, 1)) / 4)
    lod = (ct * params["lod_scale"]).clamp(0, params["lod_max"])
    share = [(1 - (lod - l).abs()).clamp(min=0) for l in range(levels)]
    num, den = torch.zeros((h, wd, 4), dtype=F64, device=DEVICE), torch.zeros_like(z)
    for ux, uy, ur in _rings():
        x, y, dist = gx + ur * ct * ux, gy + ur * ct * uy, ur * ct
        s = sum(share[l][..., None] * _bilinear(mips[l], (x + 0.5) / 2 ** l - 0.5, (y + 0.5) / 2 ** l - 0.5) for l in range(levels))
        ri = torch.where(s[..., 5] > 0, s[..., 4] / s[..., 5].clamp(min=1e-300), 0.0)
        d = sat((ri - dist) * cover + 0.5)
        num, den = num + d[..., None] * s[..., :4], den + d * s[..., 5]
    f = torch.where(den[..., None] > 0, num / den.clamp(min=1e-300)[..., None], med)
    b = (var_blur * params["var_w_recon"]).clamp(0, params["b_max"])[..., None]
    recon = torch.where(mask[..., None], med + b * (f - med), 0.0)
    # composite at full resolution
    Y, X = torch.meshgrid(torch.arange(H, device=DEVICE, dtype=F64), torch.arange(W, device=DEVICE, dtype=F64), indexing="ij")
    xh, yh = 0.5 * (X + 0.5) - 0.5, 0.5 * (Y + 0.5) - 0.5
    P = _bilinear(pp, xh, yh)
    S = _bilinear(torch.cat((recon * v, v), -1), xh, yh)
    cov = S[..., 4]
    rt = S[..., :4] / cov.clamp(min=1e-300)[..., None]
    c = _coc(cam, W, depth.to(F64).clamp(max=params["z_far_m"]))
    ws = sat((math.sqrt(2) - c.abs() + params["zof_ramp_px"] / 2) / params["zof_ramp_px"])[..., None]
    u = sat(rt[..., 3] / params["h_edge"])
    tb = torch.where(c < 0, P[..., 3], u * u * (3 - 2 * u))[..., None]
    blur = torch.where(cov[..., None] > 0, P[..., :3] + cov[..., None] * (rt[..., :3] + tb * (P[..., :3] - rt[..., :3]) - P[..., :3]),
                       P[..., :3])
    image = blur + ws * (color[..., :3].to(F64) - blur)
    return torch.cat((image, torch.ones_like(image[..., :1])), -1), new, var_blur


def exact(case, seed):
    kind, seed = case["kind"], int(seed)
    if kind == "tiles":
        s = prepare(case, seed)
        params = s["params"]
        return _dilated(_half_depth(s["depth"], s["cam"], params)[1], params)
    if case.get("lens") != "c1" or case["width"] * case["height"] > 640 * 360:
        return None
    w = _workload("c1", case["width"], case["height"], 0, seed, 1)
    if kind in ("gbuffer", "raster", "upload"):
        return _exact_gbuffer(w, Camera.from_poses(w.intr, w.poses[0]))
    if case["m"] or case["storage"] or case["blades"] or case["taa"]:
        return None
    s = prepare(case, seed)["session"]
    g, hist = s.gbufs[0], None
    for k in range(WARM + 1):
        image, hist, var = _exact_frame(w, s.cams[0], s.params, g["color"], g["depth"], k, hist)
    planes = hist.view(-1, 12)
    planes = torch.stack((planes[:, 0:4], planes[:, 4:8], planes[:, 8:12]))
    return dict(image=image, history=planes, variance=var.reshape(-1))
