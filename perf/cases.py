"""The calls whose speed this repository watches: what each one is, its inputs and its outputs.

Every case goes through the Python binding of the C-ABI (``capi``), as a program that renders
stereo pairs, trains the retrace network or builds trees does. A case is a dict of plain values;
``prepare`` makes what such a program holds before the call (scene handle, network, buffers),
``run`` makes the call, ``exact`` gives the same outputs in 64 bits from plain torch where that
is quick (brute-force ray tracing of small scenes, the network and its gradients).
"""
import math

import numpy as np
import torch

from paper_1702_01530_gb300 import capi, scenegen as sg
from paper_1702_01530_gb300.train_reproj import load_weights

DEV = "cuda"
BACKGROUND = (0.2, 0.3, 0.5)
LAYERS = ((10, 32), (32, 32), (32, 32), (32, 1))


def listed():
    return [
        # interactive preview: the 10-primitive scene at 320x240, where launches and latency count
        {"name": "render_small", "kind": "render", "scene": "small", "size": 8, "W": 320, "H": 240},
        # the benchmark's frame: 257k primitives, 4 lights, mirrors to depth 5, 1920x1080 per eye
        {"name": "render_blobs_1080p", "kind": "render", "scene": "blobs", "size": 200, "W": 1920, "H": 1080},
        # a large frame: 2.1 M triangles (a tree beyond L2), 8 lights, 3840x2160 per eye
        {"name": "render_terrain_4k", "kind": "render", "scene": "terrain", "size": 1025, "W": 3840, "H": 2160},
        # one rank's share of a pair split into bands of rows, at an odd width and offset
        {"name": "render_rows_odd", "kind": "render", "scene": "blobs", "size": 37, "W": 1367, "H": 769,
         "row0": 251, "rows": 257},
        # a server's batch: uneven requests over several resident scenes in one launch
        {"name": "batch_16", "kind": "batch", "scenes": 5, "requests": 16},
        # the retrace network on one 1080p frame, BF16
        {"name": "net_bf16_1080p", "kind": "net", "fp8": False, "images": 1, "W": 1920, "H": 1080},
        # the retrace network on eight 4K frames of a flight, FP8
        {"name": "net_fp8_8x4k", "kind": "net", "fp8": True, "images": 8, "W": 3840, "H": 2160},
        # a training step at the size the shipped weights were trained at
        {"name": "train_960x540", "kind": "train", "W": 960, "H": 540},
        # a training step on a small odd crop
        {"name": "train_251x143", "kind": "train", "W": 251, "H": 143},
        # learned reprojection of eight frames of a terrain flight, FP8 network
        {"name": "reproj_8x1080p", "kind": "reproj", "size": 513, "frames": 8, "net": "fp8", "W": 1920, "H": 1080},
        # a new scene from host arrays, its first small pair, and its release
        {"name": "create_257k", "kind": "create", "scene": "blobs", "size": 200, "W": 320, "H": 240},
        # a tree for an engine that owns its memory: 1,000,000 device-resident primitives
        {"name": "lbvh_1m", "kind": "lbvh", "spheres": 1000, "tris": 999000},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _size(rng, lo, hi):
    W = _log_int(rng, lo, hi)
    return W, max(24, int(W * rng.uniform(0.4, 0.75)))


def draw(rng):
    kind = rng.choice(("render", "render", "render", "net", "net", "train", "train", "reproj", "create", "lbvh", "batch"))
    if kind == "render":
        scene = rng.choice(("small", "polyhedra", "blobs", "terrain"))
        size = {"small": (1, 40), "polyhedra": (1, 6), "blobs": (1, 200), "terrain": (33, 1025)}[scene]
        W, H = _size(rng, 64, 3000 if scene == "terrain" else 1920)
        c = {"kind": kind, "scene": scene, "size": _log_int(rng, *size), "W": W, "H": H}
        if rng.random() < 0.25:
            c["row0"] = rng.randrange(H)
            c["rows"] = rng.randint(1, H - c["row0"])
        return c
    if kind == "net":
        W, H = _size(rng, 48, 2560)
        most = max(1, min(8, 12_000_000 // (W * H)))
        return {"kind": kind, "fp8": rng.random() < 0.5, "images": rng.randint(1, most), "W": W, "H": H}
    if kind == "train":
        W, H = _size(rng, 48, 1400)
        return {"kind": kind, "W": W, "H": H}
    if kind == "reproj":
        W, H = _size(rng, 96, 1600)
        return {"kind": kind, "size": _log_int(rng, 33, 513), "frames": rng.randint(1, 8),
                "net": rng.choice(("fp8", "bf16", "none")), "W": W, "H": H}
    if kind == "create":
        scene = rng.choice(("small", "blobs", "terrain"))
        size = {"small": (1, 40), "blobs": (1, 200), "terrain": (17, 513)}[scene]
        return {"kind": kind, "scene": scene, "size": _log_int(rng, *size), "W": 320, "H": 240}
    if kind == "lbvh":
        return {"kind": kind, "spheres": _log_int(rng, 1, 100_000), "tris": _log_int(rng, 100, 900_000)}
    return {"kind": kind, "scenes": rng.randint(1, 5), "requests": rng.randint(2, 16)}


# ------------------------------------------------------------------ inputs
def _scene(c, seed):
    """The scene of a case; another seed gives other geometry (polyhedra: another camera height)."""
    W, H, n = c["W"], c["H"], c["size"]
    if c["scene"] == "small":
        return sg.config_small(seed, W=W, H=H, n_spheres=n)
    if c["scene"] == "polyhedra":
        s = sg.config_polyhedra(n, 1 + n % 4, W=W, H=H, ground=True)
        return s.with_view(camera=sg.make_camera((0.0, 2.0 + 0.01 * (seed % 100), 0.0), (0, 0, -1), (0, 1, 0), 60.0))
    if c["scene"] == "blobs":
        return sg.config_blobs(seed, n_blobs=n, n_spheres=5 * n, box=50.0 * (n / 200.0) ** (1.0 / 3.0), W=W, H=H)
    return sg.config_terrain(seed, n_grid=n, W=W, H=H)


def _features(seed, images, W, H):
    """Network inputs with the ranges the forward warp gives: surfaces some pixels wide, a few holes."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    bw, bh = (W + 15) // 16, (H + 7) // 8

    def blocks(ch):
        low = torch.rand((images, ch, bh, bw), generator=g, device=DEV)
        return torch.nn.functional.interpolate(low, size=(bh * 8, bw * 16), mode="nearest")[:, :, :H, :W]

    f = torch.zeros((images, H, W, 16), dtype=torch.bfloat16, device=DEV)
    z = blocks(1)
    n = torch.nn.functional.normalize(2.0 * blocks(3) - 1.0, dim=1)
    f[..., 0] = (0.02 + 0.98 * z)[:, 0]
    for k in range(3):
        f[..., 1 + k] = n[:, k]
        f[..., 5 + k] = torch.rand((images, H, W), generator=g, device=DEV)
    f[..., 4] = blocks(1)[:, 0]
    f[..., 8] = (0.5 / (0.02 + z) - 1.0)[:, 0] / 16.0
    f[..., 9] = 0.7 * (blocks(1)[:, 0] < 0.1)
    f[(torch.rand((images, H, W), generator=g, device=DEV) < 0.01)] = 0
    return f


def _labels(seed, W, H):
    """1 % of the pixels to retrace, in runs as along silhouettes."""
    g = torch.Generator(device=DEV).manual_seed(seed + 1)
    low = torch.rand((1, 1, H, (W + 3) // 4), generator=g, device=DEV) < 0.01
    return low.float().repeat_interleave(4, dim=3)[0, 0, :, :W].contiguous()


def _images(n, H, W):
    return torch.empty((n, H, W, 3), dtype=torch.float32, device=DEV)


class _Batch:
    """A batch with its scenes and images; released with the object."""

    def __init__(self, case, seed):
        scenes, _ = sg.config_batch(seed, n_scenes=case["scenes"], n_requests=1)
        _, reqs = sg.config_batch(n_scenes=1, n_requests=case["requests"])   # sizes and depths do not follow the seed
        self.handles = [capi.GpuScene(s) for s in scenes]
        self.outs, items = [], []
        for r, (_, W, H, D) in enumerate(reqs):
            out = _images(2, H // 2, W // 2)
            i = r % len(scenes)
            s = scenes[i]
            items.append((self.handles[i].handle, s.camera, s.eye_sep, s.convergence, W // 2, H // 2, D, out[0], out[1]))
            self.outs.append(out)
        self.batch = capi.rt_batch_create(capi.make_requests(items))

    def __del__(self):
        if getattr(self, "batch", None):
            torch.cuda.synchronize()
            capi.rt_batch_destroy(self.batch)


def _net(case, seed, feats):
    """The shipped weights, in FP8 with scales calibrated on these features when the case says so."""
    net = capi.Net(load_weights()[0])
    if case.get("fp8") or case.get("net") == "fp8":
        capi.rt_net_calibrate_fp8(net.handle, [feats[0].contiguous()], feats.shape[2], feats.shape[1])
    return net


def prepare(case, seed):
    k = case["kind"]
    st = {"case": case}
    if k in ("render", "reproj"):
        c = dict(case, scene=case.get("scene", "terrain"))
        s = _scene(c, seed)
        st["scene"], st["gpu"] = s, capi.GpuScene(s)
    if k == "render":
        st["out"] = _images(2, case.get("rows", case["H"]), case["W"])
    elif k == "create":
        st["scene"], st["out"] = _scene(case, seed), _images(2, case["H"], case["W"])
    elif k == "batch":
        st["batch"] = _Batch(case, seed)
    elif k == "net":
        st["feat"] = _features(seed, case["images"], case["W"], case["H"])
        st["net"] = _net(case, seed, st["feat"])
        st["prob"] = torch.empty((case["images"], case["H"], case["W"]), dtype=torch.float32, device=DEV)
    elif k == "train":
        st["feat"] = _features(seed, 1, case["W"], case["H"])
        st["label"] = _labels(seed, case["W"], case["H"])
        st["net"] = capi.Net(sg.net_params_he(seed))
        st["grads"] = torch.empty(capi.RT_NET_PARAMS, dtype=torch.float32, device=DEV)
    elif k == "reproj":
        st["cams"] = sg.terrain_cameras(seed, n_frames=case["frames"])
        if case["net"] != "none":
            st["net"] = _net(case, seed, _features(seed, 1, 960, 540))
        st["L"], st["R"] = _images(case["frames"], case["H"], case["W"]), _images(case["frames"], case["H"], case["W"])
    elif k == "lbvh":
        g = torch.Generator(device=DEV).manual_seed(seed)
        ns, nt = case["spheres"], case["tris"]
        c = torch.rand((ns + nt, 3), generator=g, device=DEV) * 100.0 - 50.0
        c[:, 1] *= 0.2                                    # a scene wider than it is high
        st["sph"] = torch.cat([c[:ns], 0.05 + 0.45 * torch.rand((ns, 1), generator=g, device=DEV),
                               torch.zeros((ns, 1), device=DEV)], 1).contiguous()
        v = c[ns:, None, :] + torch.randn((nt, 3, 3), generator=g, device=DEV) * 0.1
        st["tri"] = torch.cat([v.reshape(nt, 9), torch.zeros((nt, 1), device=DEV)], 1).contiguous()
        n = ns + nt
        st["nodes"] = torch.empty((max(n - 1, 1), 16), dtype=torch.int32, device=DEV)
        st["prims"] = torch.empty((n, 12), dtype=torch.int32, device=DEV)
        st["keys"] = torch.empty(n, dtype=torch.int64, device=DEV)
        st["parent"] = torch.empty(2 * n - 1, dtype=torch.int32, device=DEV)
    return st


def run(st):
    c = st["case"]
    k = c["kind"]
    if k == "render":
        s, out = st["scene"], st["out"]
        if "rows" in c:
            capi.rt_render_stereo_rows(st["gpu"].handle, s.camera, s.eye_sep, s.convergence, s.W, s.H, s.max_depth,
                                       c["row0"], c["rows"], out[0], out[1])
        else:
            capi.rt_render_stereo(st["gpu"].handle, s.camera, s.eye_sep, s.convergence, s.W, s.H, s.max_depth,
                                  out[0], out[1])
        return out
    if k == "create":
        g = capi.GpuScene(st["scene"])
        g.render(out=st["out"])
        capi.rt_sync_status(g.handle)
        g.close()
        return st["out"]
    if k == "batch":
        capi.rt_batch_launch(st["batch"].batch)
        return st["batch"].outs
    if k == "net":
        if c["images"] == 1:
            capi.rt_net_forward(st["net"].handle, st["feat"], c["W"], c["H"], st["prob"])
        else:
            capi.rt_net_forward_images(st["net"].handle, st["feat"], c["images"], c["W"], c["H"], st["prob"])
        return st["prob"]
    if k == "train":
        # the training loop reads the loss of a few steps only
        capi.rt_net_train_step(st["net"].handle, st["feat"], st["label"], c["W"], c["H"], 1e-3, want_loss=False,
                               grads=st["grads"])
        return st["grads"]
    if k == "reproj":
        s = st["scene"]
        net = st["net"].handle if "net" in st else None
        capi.rt_render_stereo_reproj_frames(st["gpu"].handle, st["cams"], s.eye_sep, s.convergence, s.W, s.H,
                                            s.max_depth, net, 0.1, st["L"], st["R"])
        return st["L"], st["R"]
    capi.rt_build_lbvh_noalloc(st["sph"], c["spheres"], st["tri"], c["tris"], st["nodes"], st["prims"], st["keys"],
                               st["parent"])
    return st["nodes"], st["prims"], st["keys"], st["parent"]


# ------------------------------------------------------------ work and errors
def _prims(c):
    n = c["size"]
    return {"small": (n, 2), "polyhedra": (0, 12 * n + 60), "blobs": (5 * n, 1280 * n),
            "terrain": (10000, 2 * (n - 1) ** 2)}[c.get("scene", "terrain")]


def _trace_work(ns, nt, lights, pixels):
    """Both eyes: a primary ray, a shadow ray to half of the lights; a root-to-leaf walk (40 operations
    a level) and a triangle test each, and the shading; scene records read once, images written once."""
    rays = 2 * pixels * (1 + 0.5 * lights)
    return {"bytes": 20 * ns + 40 * nt + 24 * pixels,
            "flops": rays * (40 * math.ceil(math.log2(ns + nt + 1)) + 41 + 40)}


def work(case):
    k = case["kind"]
    lights = {"small": 1, "polyhedra": 2, "blobs": 4, "terrain": 8}
    if k in ("render", "create"):
        pixels = case["W"] * case.get("rows", case["H"])
        return _trace_work(*_prims(case), lights[case["scene"]], pixels)
    if k == "batch":
        scenes, reqs = case["scenes"], case["requests"]
        nt = sum(1280 * max(1, round(1e3 * 2000.0 ** (i / max(1, scenes - 1)) / 1280.0)) for i in range(scenes))
        return _trace_work(nt // 256, nt, 4, reqs * 710_000)   # a quarter of the mean of 640x360 .. 3840x2160
    P = case.get("W", 0) * case.get("H", 0) * case.get("images", 1)
    macs = sum(9 * ci * co for ci, co in LAYERS)
    if k == "net":
        return {"bytes": P * (32 + 4) + 4 * capi.RT_NET_PARAMS, "flops": 2 * P * macs}
    if k == "train":    # forward, weight gradients, data gradients of all but the first layer
        return {"bytes": P * (32 + 4) + 4 * 8 * capi.RT_NET_PARAMS, "flops": 2 * P * (3 * macs - 9 * 10 * 32)}
    if k == "reproj":   # one eye of each frame traced; the network
        ns, nt = _prims(case)
        P *= case["frames"]
        w = _trace_work(ns, nt, 8, P)
        return {"bytes": w["bytes"], "flops": w["flops"] / 2 + (2 * P * macs if case["net"] != "none" else 0)}
    n = case["spheres"] + case["tris"]
    return {"bytes": 20 * case["spheres"] + 40 * case["tris"] + n * (64 + 48 + 8 + 8), "flops": n * 100}


def tolerance(case):
    k = case["kind"]
    if k == "lbvh":
        return "exact"                       # an integer key order and boxes of stated rounding
    if k in ("render", "create", "batch"):
        # FP32 rays are 5e-7 off 64-bit ones until a shadow or silhouette edge falls on the other side of
        # a pixel's ray: then that pixel changes wholly, and a few of them in a small image give 1e-3
        return {"rel": 2e-3, "max": 0.99}
    if k == "reproj":
        # the same, and pixels whose retrace probability lies next to the threshold
        return {"rel": 5e-3, "max": 0.99}
    if k == "net":
        # four times what BF16 activations (5e-3) and E4M3 ones (6e-2, so capped) differ from 64 bits by
        return {"rel": 2.9e-2, "max": 0.99} if case["fp8"] else {"rel": 2e-2, "max": 0.5}
    return {"rel": 1.2e-2, "max": 0.5}       # gradients through four layers of BF16 activations: 3e-3 off


# ------------------------------------------------------------------ exact
def exact(case, seed):
    if case["kind"] in ("render", "create"):
        ns, nt = _prims(case)
        if ns + nt > 200 or case["W"] * case["H"] * (ns + nt) > 1e8:
            return None
        s = _scene(case, seed)
        return _trace(s, case.get("row0", 0), case.get("rows", case["H"]))
    if case["kind"] == "net":
        with torch.no_grad():
            w = _split(torch.tensor(load_weights()[0], dtype=torch.float64, device=DEV))
            feat = _features(seed, case["images"], case["W"], case["H"])
            return torch.stack([torch.sigmoid(_logits(f, w)) for f in feat])
    if case["kind"] == "train":
        p = torch.tensor(sg.net_params_he(seed), dtype=torch.float64, device=DEV, requires_grad=True)
        y = _labels(seed, case["W"], case["H"]).double()
        z = _logits(_features(seed, 1, case["W"], case["H"])[0], _split(p))
        torch.nn.functional.binary_cross_entropy_with_logits(z, y).backward()
        return p.grad
    return None


def _split(p):
    out, at = [], 0
    for ci, co in LAYERS:
        out.append((p[at:at + co * ci * 9].view(co, ci, 3, 3), p[at + co * ci * 9:at + co * ci * 9 + co]))
        at += co * ci * 9 + co
    return out


def _logits(feat, weights):
    """H x W logits of one image: each layer as nine shifted matrix products in float64."""
    x = feat[..., :10].double()
    H, W = x.shape[:2]
    for i, (w, b) in enumerate(weights):
        xp = torch.nn.functional.pad(x, (0, 0, 1, 1, 1, 1))
        y = b
        for ky in range(3):
            for kx in range(3):
                y = y + xp[ky:ky + H, kx:kx + W] @ w[:, :, ky, kx].t()
        x = torch.relu(y) if i < 3 else y
    return x[..., 0]


def _closest(o, d, sph, tri):
    """Nearest hit parameter (inf on a miss) and its primitive, lower ids first among equals."""
    ts = []
    if len(sph):
        oc = o[:, None] - sph[None, :, :3]
        b = (oc * d[:, None]).sum(-1)
        disc = b * b - (oc * oc).sum(-1) + sph[:, 3] ** 2
        sq = disc.clamp(min=0).sqrt()
        near, far = -b - sq, -b + sq
        t = torch.where(near > 0, near, far)
        ts.append(torch.where((disc >= 0) & (t > 0), t, math.inf))
    if len(tri):
        v0, e1, e2 = tri[:, 0], tri[:, 1] - tri[:, 0], tri[:, 2] - tri[:, 0]
        dd, e1, e2 = torch.broadcast_tensors(d[:, None], e1[None], e2[None])
        pv = torch.linalg.cross(dd, e2)
        det = (e1 * pv).sum(-1)
        tv = o[:, None] - v0[None]
        qv = torch.linalg.cross(tv, e1)
        u, v, t = (tv * pv).sum(-1) / det, (dd * qv).sum(-1) / det, (e2 * qv).sum(-1) / det
        ok = (det != 0) & (u >= 0) & (v >= 0) & (u + v <= 1) & (t > 0)
        ts.append(torch.where(ok, t, math.inf))
    return torch.cat(ts, 1).min(1)


def _unit(v):
    return v / v.norm(dim=-1, keepdim=True)


def _trace(s, row0, rows):
    """Both eyes of the scene's rows in float64, every primitive tested by every ray."""
    f64 = lambda a: torch.tensor(np.asarray(a, np.float64), device=DEV)   # noqa: E731
    sph = torch.cat([f64(s.spheres["center"]).reshape(-1, 3), f64(s.spheres["radius"])[:, None]], 1)
    tri = torch.stack([f64(s.triangles[k]).reshape(-1, 3) for k in ("v0", "v1", "v2")], 1)
    mat = torch.tensor(np.concatenate([s.spheres["material"], s.triangles["material"]]).astype(np.int64), device=DEV)
    alb, refl = f64(s.materials["albedo"]), f64(s.materials["reflectivity"])
    lpos, lint = f64(s.lights["position"]), f64(s.lights["intensity"])
    eye, up = f64(s.camera["eye"]), f64(s.camera["up"])
    fwd = _unit(f64(s.camera["forward"]))
    right = _unit(torch.linalg.cross(fwd, up))
    up = torch.linalg.cross(right, fwd)
    tan = math.tan(math.radians(float(s.camera["vfov_deg"])) / 2)
    j, i = torch.meshgrid(torch.arange(row0, row0 + rows, device=DEV), torch.arange(s.W, device=DEV), indexing="ij")
    nx = ((2 * (i.double() + 0.5) / s.W - 1) * tan * s.W / s.H).reshape(-1, 1)
    ny = ((1 - 2 * (j.double() + 0.5) / s.H) * tan).reshape(-1, 1)
    aim = eye + float(np.float32(s.convergence)) * (fwd + nx * right + ny * up)
    half = 0.5 * float(np.float32(s.eye_sep))
    images = []
    for side in (-1.0, 1.0):
        o = eye + side * half * right
        parts = [_shade(o.expand_as(a), _unit(a - o), sph, tri, mat, alb, refl, lpos, lint, s.max_depth)
                 for a in aim.split(1 << 15)]
        images.append(torch.cat(parts).clamp(0, 1).reshape(rows, s.W, 3))
    return torch.stack(images)


def _shade(o, d, sph, tri, mat, alb, refl, lpos, lint, max_depth):
    colour = torch.zeros_like(o)
    weight = torch.ones(len(o), 1, dtype=o.dtype, device=o.device)
    live = torch.arange(len(o), device=o.device)
    for depth in range(max_depth + 1):
        t, k = _closest(o, d, sph, tri)
        miss = torch.isinf(t)
        colour[live[miss]] += weight[miss] * torch.tensor(BACKGROUND, dtype=o.dtype, device=o.device)
        live, o, d, t, k, weight = live[~miss], o[~miss], d[~miss], t[~miss], k[~miss], weight[~miss]
        if not len(live):
            break
        p = o + d * t[:, None]
        n = torch.empty_like(p)
        is_s = k < len(sph)
        n[is_s] = (p[is_s] - sph[k[is_s], :3]) / sph[k[is_s], 3:]
        v = tri[k[~is_s] - len(sph)]
        n[~is_s] = _unit(torch.linalg.cross(v[:, 1] - v[:, 0], v[:, 2] - v[:, 0]))
        n = torch.where((n * d).sum(-1, keepdim=True) > 0, -n, n)
        eps = 1e-4 * p.abs().amax(1, keepdim=True).clamp(min=1.0)
        p = p + n * eps
        light = torch.full_like(t, 0.1)
        for lp, li in zip(lpos, lint):
            lv = lp - p
            dist = lv.norm(dim=-1)
            lh = lv / dist[:, None]
            ndl = (n * lh).sum(-1)
            free = _closest(p, lh, sph, tri)[0] >= dist - eps[:, 0]
            light = light + torch.where((ndl > 0) & free, li * ndl, 0.0)
        r = refl[mat[k]][:, None]
        colour[live] += weight * (1 - r) * alb[mat[k]] * light[:, None]
        go = r[:, 0] > 0
        o, d, weight, live = p[go], _unit(d[go] - 2 * (d[go] * n[go]).sum(-1, keepdim=True) * n[go]), (weight * r)[go], live[go]
        if not len(live):
            break
    return colour
