"""Performance cases of the fusion path, each one pass through a public entry point.

What the cases stand for:

* ``frame_2x160x120_f32``: the smallest rig of the test suite (two float32 sensors), one
  ``fuse`` call a frame: latency and launches count.
* ``graph_4x640x480``: an ordinary rig whose frames land in fixed buffers, replayed from a
  recorded call (``FuseFlow.graph``).
* ``ragged_5_screened_f32``: cameras of different, odd sizes with float32 depth and the depth
  screen set (nothing aligned, tiles and rows cut).
* ``frame_8x1280x720``: the benchmark rig, one ``fuse`` call a frame.
* ``batch_4_of_8x1280x720``: the benchmark as configured, four frames in one batched launch
  replayed from a recorded graph.
* ``top3_8x1280x720``: the top-k variant on the benchmark rig.
* ``frame_16x1024`` and ``frame_32x1024``: the large rigs of the scaling sweep (sparse far walls,
  dense near objects; millions of cells).
* ``points_8x1280x720``: point-wise fusion without the spatial hash.
* ``confidence_8x1280x720``: the confidence producer for sensors without a confidence image.
* ``mc_error_200k``: the multi-camera depth consistency error of a cloud.
* ``host_4x640x480``: host images in, host cloud out, one synchronous call.

Drawn cases take the same kinds over 2..24 cameras, widths 160..1920, odd sizes, both depth
formats, mixed resolutions, top-k 1..7 and 2..6 views.

Inputs are rendered on the GPU from the seed alone: a ground plane or a room with seeded
primitives, depth noise 0.0015 z^2, 1 % flying pixels at depth edges, 1 % missing samples,
grazing-angle confidence and lattice colours.
"""
import math

import numpy as np
import torch

from paper_2602_01035_gb300 import fuseflow as F
from paper_2602_01035_gb300 import scenes as S

TAU, SIGMA_M, S0_M, MAX_LEVEL, N_MIN, BIAS = 0.6, 0.03, 0.32, 4, 32, 1 << 19
MAX_PX = 32 * 1024 * 1024


def _case(name, kind, layout, cams, w, h, **more):
    c = {"kind": kind, "layout": layout, "cams": cams, "w": w, "h": h, "fmt": "u16", "mixed": False,
         "k_views": 4, "top_k": 0, "screen": False, "frames": 1, "points": 0}
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        _case("frame_2x160x120_f32", "frame", "ring", 2, 160, 120, fmt="f32"),
        _case("graph_4x640x480", "graph", "ring", 4, 640, 480),
        _case("ragged_5_screened_f32", "frame", "hemi", 5, 651, 483, fmt="f32", mixed=True, screen=True),
        _case("frame_8x1280x720", "frame", "hemi", 8, 1280, 720),
        _case("batch_4_of_8x1280x720", "batch", "hemi", 8, 1280, 720, frames=4),
        _case("top3_8x1280x720", "frame", "hemi", 8, 1280, 720, top_k=3),
        _case("frame_16x1024", "frame", "sphere", 16, 1024, 1024),
        _case("frame_32x1024", "frame", "sphere", 32, 1024, 1024),
        _case("points_8x1280x720", "points", "hemi", 8, 1280, 720),
        _case("confidence_8x1280x720", "confidence", "hemi", 8, 1280, 720),
        _case("mc_error_200k", "mc", "hemi", 8, 1280, 720, points=200_000),
        _case("host_4x640x480", "host", "ring", 4, 640, 480),
    ]


def draw(rng):
    kind = rng.choice(["frame", "frame", "frame", "graph", "batch", "top_k", "points", "confidence",
                       "screen", "mc", "host"])
    w = int(round(math.exp(rng.uniform(math.log(160), math.log(1920)))))
    w = w // 8 * 8 if rng.random() < 0.5 else w
    h = max(90, int(w * rng.uniform(0.5, 1.0)))
    cams = int(round(math.exp(rng.uniform(math.log(2), math.log(24)))))
    frames = rng.randint(2, 8) if kind == "batch" else 1
    limit = MAX_PX // 4 if kind == "host" else MAX_PX // 2
    while cams * w * h * frames > limit:
        if frames > 2:
            frames -= 1
        elif cams > 2:
            cams -= 1
        else:
            w, h = w * 3 // 4, max(90, h * 3 // 4)
    return _case(None, "frame" if kind == "top_k" else kind, rng.choice(["ring", "hemi", "sphere"]), cams, w, h,
                 fmt=rng.choice(["u16", "u16", "f32"]), mixed=rng.random() < 0.25,
                 k_views=rng.choice([2, 3, 4, 4, 4, 6]), top_k=rng.randint(1, 7) if kind == "top_k" else 0,
                 screen=kind == "screen" or (kind in ("frame", "graph") and rng.random() < 0.2), frames=frames,
                 points=int(math.exp(rng.uniform(math.log(1000), math.log(1_000_000)))) if kind == "mc" else 0)


# ------------------------------------------------------------------------------------ inputs
def _rig(case):
    n, w0, h0 = case["cams"], case["w"], case["h"]
    cams = []
    for k in range(n):
        w, h = (w0 * 5 // 8 + 1, h0 * 3 // 4) if case["mixed"] and k % 2 else (w0, h0)
        if case["layout"] == "sphere":         # inside a room, looking at the centre
            z = 1.0 - 2.0 * (k + 0.5) / n
            a, r = math.pi * (3.0 - math.sqrt(5.0)) * k, math.sqrt(max(0.0, 1.0 - z * z))
            c, f = 5.0 * np.array([r * math.cos(a), r * math.sin(a), z]), 0.5 * w
        elif case["layout"] == "hemi":
            e, a = math.radians(20.0 + 40.0 * k / max(1, n - 1)), 2.0 * math.pi * k / n
            c, f = 4.0 * np.array([math.cos(e) * math.cos(a), math.cos(e) * math.sin(a), math.sin(e)]), 0.703 * w
        else:
            a = 2.0 * math.pi * (k / n if n > 3 else k / 6) + 0.7
            c, f = np.array([3.0 * math.cos(a), 3.0 * math.sin(a), 1.5]), 0.82 * w
        cams.append(S.look_at(c, (0, 0, 0), f, f, w / 2, h / 2, w, h))
    return S.Rig(cams, case["fmt"], 1.0 if case["fmt"] == "f32" else 0.001)


def _primitives(case, rng):
    if case["layout"] == "sphere":
        prims = [("room", np.full(3, -8.0), np.full(3, 8.0)), ("box", np.full(3, -0.6), np.full(3, 0.6))]
        for _ in range(8):
            v = rng.normal(size=3)
            prims.append(("sphere", 4.0 * v / np.linalg.norm(v), rng.uniform(0.2, 0.5)))
        return prims
    prims = [("plane",)]
    for k in range(16):
        rad, ang, size = rng.uniform(0.2, 2.8), rng.uniform(0, 2 * np.pi), rng.uniform(0.1, 0.6)
        x, y, half = rad * math.cos(ang), rad * math.sin(ang), size / 2
        prims.append(("sphere", np.array([x, y, half]), half) if k % 2 else
                     ("box", np.array([x - half, y - half, 0.0]), np.array([x + half, y + half, size])))
    return prims


def _cast(o, d, prims):
    """Nearest z-depth along the rays o + t d (camera-z of d is 1) and the normal's cosine."""
    inf = torch.full(d.shape[:2], math.inf, device=d.device)
    z, cos = inf.clone(), torch.zeros_like(inf)
    length = d.norm(dim=2)
    for p in prims:
        if p[0] == "plane":
            t = -o[2] / d[..., 2]
            t = torch.where(t > 1e-3, t, inf)
            c = d[..., 2].abs() / length
        elif p[0] == "sphere":
            oc = o - torch.as_tensor(p[1], dtype=torch.float32, device=d.device)
            a, b, q = (d * d).sum(2), (d * oc).sum(2), (oc * oc).sum() - p[2] ** 2
            disc = b * b - a * q
            t = (-b - disc.clamp(min=0).sqrt()) / a
            t = torch.where((disc >= 0) & (t > 1e-3), t, inf)
            c = (disc.clamp(min=0).sqrt() / (length * p[2])).clamp(max=1.0)
        else:
            lo, hi = (torch.as_tensor(v, dtype=torch.float32, device=d.device) for v in p[1:3])
            t1, t2 = (lo - o) / d, (hi - o) / d
            near, far = torch.minimum(t1, t2), torch.maximum(t1, t2)
            (tn, an), (tf, af) = near.max(2), far.min(2)
            if p[0] == "room":
                t, axis = torch.where(tf > 1e-3, tf, inf), af
            else:
                t, axis = torch.where((tf >= tn) & (tn > 1e-3), tn, inf), an
            c = d.gather(2, axis[..., None])[..., 0].abs() / length
        closer = t < z
        z, cos = torch.where(closer, t, z), torch.where(closer, c, cos)
    return z, cos


def _images(case, rig, seed):
    """(depth, conf, rgb): per-camera CUDA images of one seeded frame."""
    rng = np.random.default_rng(seed)
    prims = _primitives(case, rng)
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed * 7919 + 13)
    out = ([], [], [])
    for cam in rig.cameras:
        x = (torch.arange(cam.width, device=dev, dtype=torch.float32) - cam.cx) / cam.fx
        y = (torch.arange(cam.height, device=dev, dtype=torch.float32) - cam.cy) / cam.fy
        ray = torch.stack([x[None, :].expand(cam.height, -1), y[:, None].expand(-1, cam.width),
                           torch.ones(cam.height, cam.width, device=dev)], 2)
        d = ray @ torch.as_tensor(cam.R, dtype=torch.float32, device=dev)
        o = torch.as_tensor(cam.centre, dtype=torch.float32, device=dev)
        z, cos = _cast(o, d, prims)
        hit = (z < 60.0)
        z = torch.where(hit, z, torch.zeros_like(z))
        lattice = torch.floor((o + z[..., None] * d) * 100.0 + 0.5).to(torch.int64)
        code = (lattice * torch.tensor([73856093, 19349663, 83492791], device=dev)).sum(2)
        code = (code ^ (code >> 13)) * 0x5BD1E995 & 0xFFFFFFFF
        rgb = torch.stack([(code >> s) & 255 for s in (0, 8, 16)], 2) * hit[..., None]
        pool = torch.nn.functional.max_pool2d
        zmax = pool(z[None, None], 3, 1, 1)[0, 0]
        zmin = -pool(torch.where(hit, -z, torch.full_like(z, -1e9))[None, None], 3, 1, 1)[0, 0]
        edge = hit & (zmax - zmin > 0.1)
        r = torch.rand(4, *z.shape, generator=gen, device=dev)
        zn = z + torch.randn(z.shape, generator=gen, device=dev) * 0.0015 * z * z
        share = min(1.0, 0.01 * z.numel() / max(1, int(edge.sum())))
        zn = torch.where(edge & (r[0] < share), zmin + r[1] * (zmax - zmin), zn)
        zn = torch.where(hit & (zn > 0) & (r[2] >= 0.01), zn, torch.zeros_like(zn))
        conf = 1.0 - 0.5 * (1.0 - cos * cos).clamp(min=0).sqrt() + (r[3] - 0.5) * 0.1
        conf = torch.where(hit, conf.clamp(0.0, 1.0), torch.zeros_like(conf))
        if case["fmt"] == "u16":
            depth = (zn * 1000.0).round().clamp(0, 65535).to(torch.int32).to(torch.uint16)
        else:
            depth = zn
        out[0].append(depth.contiguous())
        out[1].append(conf.contiguous())
        out[2].append(rgb.to(torch.uint8).contiguous())
    return out


def _points(case, rig, images, seed):
    """World points near the observed surfaces: samples of the depth images, jittered by 5 mm."""
    n, dev = case["points"], torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed * 31 + 7)
    parts = []
    for k, cam in enumerate(rig.cameras):
        m = (n - k + len(rig.cameras) - 1) // len(rig.cameras)
        x = torch.randint(0, cam.width, (m,), generator=gen, device=dev)
        y = torch.randint(0, cam.height, (m,), generator=gen, device=dev)
        z = images[0][k].to(torch.float32)[y, x] * rig.depth_scale
        p = torch.stack([(x - cam.cx) / cam.fx * z, (y - cam.cy) / cam.fy * z, z], 1).to(torch.float64)
        p = (p - torch.as_tensor(cam.t, device=dev)) @ torch.as_tensor(cam.R, device=dev)
        parts.append(p.to(torch.float32))
    pts = torch.cat(parts)[:n]
    return (pts + 0.005 * torch.randn(pts.shape, generator=gen, device=dev)).contiguous()


# ------------------------------------------------------------------------------------ passes
class _State:
    pass


class _Array:
    """A context-owned device array that keeps its context alive as long as a view of it lives."""

    def __init__(self, owner, ptr, shape, typestr):
        self.owner = owner
        self.__cuda_array_interface__ = {"shape": shape, "typestr": typestr, "data": (int(ptr), False), "version": 3,
                                         "strides": None}


def _params(case):
    p = {"k_views": case["k_views"], "top_k": case["top_k"]}
    if case["screen"]:
        p.update(screen_min_m=0.3, screen_max_m=12.0, screen_edge_rel=0.03)
    return p


def _views(ff):
    """The context's whole output arrays (entries past the frame's cells stay zero)."""
    c, n = F.fuseflow_get_cloud(ff.ctx), ff.capacity
    arrays = {"pos": (c.pos, (n, 3), "<f4"), "rgb": (c.rgb, (n, 3), "<f4"), "weight": (c.weight, (n,), "<f4"),
              "count": (c.count, (n,), "<i4"), "rep": (c.rep, (n,), "<i4"), "key": (c.key, (n,), "<i8"),
              "pixels_and_cells": (c.stats, (4,), "<i8"), "extent": (c.stats + 32, (6,), "<f4"),
              "error_and_coarse": (c.stats + 56, (2,), "<i4")}
    return {k: torch.as_tensor(_Array(ff, *v), device="cuda") for k, v in arrays.items()}


def prepare(case, seed):
    s, kind = _State(), case["kind"]
    s.kind, s.rig = kind, _rig(case)
    s.frames = [_images(case, s.rig, seed * 64 + f) for f in range(case["frames"])]
    s.ff = [F.FuseFlow(s.rig, **_params(case)) for _ in s.frames]
    dev, n_px = torch.device("cuda"), s.ff[0].n_pixels
    depth, conf, rgb = s.frames[0]
    if kind in ("frame", "graph", "batch"):
        s.out = [_views(ff) for ff in s.ff]
        if kind == "graph":
            s.graph = s.ff[0].graph(depth, conf, rgb)
        elif kind == "batch":
            s.batch = F.Batch(s.ff)
            s.graph = s.batch.graph(s.frames)
    elif kind == "points":
        s.out = {"pos": torch.zeros(n_px, 3, device=dev), "weight": torch.zeros(n_px, device=dev),
                 "rgb": torch.zeros(n_px, 3, dtype=torch.uint8, device=dev)}
    elif kind == "confidence":
        s.out = [torch.zeros_like(c) for c in conf]
    elif kind == "screen":
        s.out = [torch.zeros_like(d) for d in depth]
    elif kind == "mc":
        s.points = _points(case, s.rig, s.frames[0], seed)
        s.err = torch.zeros(len(s.points), device=dev)
        s.seen = torch.zeros(len(s.points), dtype=torch.int32, device=dev)
    else:
        s.host = [[t.cpu().pin_memory() for t in part] for part in s.frames[0]]
        cap = s.ff[0].capacity
        s.out = {"pos": torch.zeros(cap, 3), "rgb": torch.zeros(cap, 3), "weight": torch.zeros(cap),
                 "count": torch.zeros(cap, dtype=torch.int32), "rep": torch.zeros(cap, dtype=torch.int32),
                 "key": torch.zeros(cap, dtype=torch.int64)}
        s.out = {k: v.pin_memory() for k, v in s.out.items()}
    return s


def _ptrs(tensors):
    return [t.data_ptr() for t in tensors]


def run(s):
    depth, conf, rgb = s.frames[0]
    if s.kind == "frame":
        s.ff[0].fuse(depth, conf, rgb)
        return s.out
    if s.kind in ("graph", "batch"):
        s.graph.launch()
        return s.out
    stream = torch.cuda.current_stream().cuda_stream
    if s.kind == "points":
        F.fuseflow_fuse_points(s.ff[0].ctx, _ptrs(depth), _ptrs(conf), _ptrs(rgb), s.out["pos"].data_ptr(),
                               s.out["weight"].data_ptr(), s.out["rgb"].data_ptr(), stream, counts=False)
        return s.out
    if s.kind == "confidence":
        F.fuseflow_confidence(s.ff[0].ctx, _ptrs(depth), _ptrs(s.out), stream)
        return s.out
    if s.kind == "screen":
        F.fuseflow_screen_depth(s.ff[0].ctx, _ptrs(depth), _ptrs(s.out), stream)
        return [t.view(torch.int16) if t.dtype == torch.uint16 else t for t in s.out]
    if s.kind == "mc":
        mc, used = F.fuseflow_mc_error(s.ff[0].ctx, s.points.data_ptr(), len(s.points), _ptrs(depth),
                                       s.err.data_ptr(), s.seen.data_ptr(), stream)
        return {"mc": mc, "used": used, "err": s.err, "seen": s.seen}
    o = s.out
    status, st = F.fuseflow_fuse_frame_host(s.ff[0].ctx, *[_ptrs(p) for p in s.host],
                                            *[o[k].data_ptr() for k in ("pos", "rgb", "weight", "count", "rep", "key")],
                                            stream)
    return {"status": status, "cells": st.n_cells, "gated": st.n_gated, "coarse": st.n_coarse,
            "extent": np.array(st.bbox[:], dtype=np.float32), **o}


# ------------------------------------------------------------------------------------ claims
def work(case):
    """Inputs once (depth 2 or 4 B, confidence 4 B, colour 3 B a pixel) and outputs once; about
    half the pixels pass the gate and 20 of them share a cell of 44 B.  Operations: back-projection,
    weight and cell sums (about 40) and 30 per other view and gated pixel."""
    rig = _rig(case)
    px, d = rig.n_pixels * case["frames"], 2 if case["fmt"] == "u16" else 4
    k1 = min(case["k_views"], case["cams"]) - 1
    if case["kind"] == "confidence":
        return {"bytes": px * (d + 4), "flops": 60 * px}
    if case["kind"] == "screen":
        return {"bytes": px * 2 * d, "flops": 15 * px}
    if case["kind"] == "points":
        return {"bytes": px * (d + 7 + 19), "flops": px // 2 * (30 + 30 * k1)}
    if case["kind"] == "mc":
        return {"bytes": case["points"] * (20 + case["cams"] * d), "flops": case["points"] * case["cams"] * 25}
    return {"bytes": px * (d + 7) + px // 40 * 44, "flops": px // 2 * (40 + 30 * k1)}


def tolerance(case):
    """Counts, keys, representatives and bytes are the same.  Fused values are float32 results of
    exact integer sums of float32 terms: against 64 bits they measure 0.3e-7 to 1.1e-7, and a sum
    over another tiling moves them by less.  The consistency error picks each point's pixel in
    float32: per point it is compared only between float32 evaluations."""
    if case["kind"] == "screen":
        return "exact"
    return {"rel": 5e-7}


# ------------------------------------------------------------------------------------ 64 bits
def _f32(v):
    return v.to(torch.float32).to(torch.float64)


def _neighbours(rig, k1):
    out = []
    for i, a in enumerate(rig.cameras):
        got = []
        for j, b in enumerate(rig.cameras):
            if j != i:
                cos = a.R[2] @ b.R[2] / np.linalg.norm(a.R[2]) / np.linalg.norm(b.R[2])
                got.append((round(math.acos(max(-1.0, min(1.0, cos))), 9),
                            round(float(np.linalg.norm(a.centre - b.centre)), 9), j))
        out.append([j for _, _, j in sorted(got)[:k1]])
    return out


def _exact_screen(rig, depth):
    out = []
    for d in depth:
        z = d.to(torch.float32)
        lo, hi = np.float32(0.3 / rig.depth_scale), np.float32(12.0 / rig.depth_scale)
        fine = (z > 0) & torch.isfinite(z) & (z >= float(lo)) & (z <= float(hi))
        thr, keep = z * float(np.float32(0.03)), fine.clone()
        pad, ok = torch.nn.functional.pad(z, (1, 1, 1, 1)), torch.nn.functional.pad(fine, (1, 1, 1, 1))
        h, w = z.shape
        for dy, dx in ((0, 1), (2, 1), (1, 0), (1, 2)):
            keep &= ~(ok[dy:dy + h, dx:dx + w] & ((z - pad[dy:dy + h, dx:dx + w]).abs() > thr))
        out.append(torch.where(keep, z, torch.zeros_like(z)))
    return out


def _exact_points(case, rig, images):
    """Per camera: gate, index, point (metres, 64 bits), cell coordinate r of the float32 point,
    exponent e, confidence, colour of the gated pixels.  The cell of a point is that of its
    float32 position, as a point on a cell's face belongs to either side; all else is 64 bits."""
    depth = _exact_screen(rig, images[0]) if case["screen"] else images[0]
    u, k1 = rig.depth_scale, min(case["k_views"], case["cams"]) - 1
    near, dev, off = _neighbours(rig, k1), torch.device("cuda"), 0
    for i, cam in enumerate(rig.cameras):
        z = depth[i].to(torch.float64).reshape(-1)
        conf = images[1][i].reshape(-1)
        valid = (z > 0) & torch.isfinite(z)
        idx = torch.nonzero(valid & (conf > float(np.float32(TAU))))[:, 0]
        z, c = z[idx], conf[idx].to(torch.float64)
        x, y = idx % cam.width, torch.div(idx, cam.width, rounding_mode="floor")
        rx, ry = (x.double() - cam.cx) / cam.fx, (y.double() - cam.cy) / cam.fy
        p = torch.stack([z * rx, z * ry, z], 1) * u
        R, t = torch.as_tensor(cam.R, device=dev), torch.as_tensor(cam.t, device=dev)
        world = (p - t) @ R
        q = [_f32(_f32(z) * _f32(rx)), _f32(_f32(z) * _f32(ry)), _f32(z)]
        cen = np.asarray(cam.centre) / u
        r = []
        for a in range(3):
            v = torch.full_like(z, float(np.float32(cen[a])))
            for b in (2, 1, 0):
                v = _f32(float(np.float32(cam.R[b, a])) * q[b] + v)
            r.append(_f32(v * float(np.float32(u / S0_M))))
        e = torch.zeros_like(z)
        for j in near[i]:
            J = rig.cameras[j]
            rel = torch.as_tensor(J.R @ cam.R.T, device=dev)
            a = p @ rel.T + (torch.as_tensor(J.t, device=dev) - rel @ t)
            az = a[:, 2].clamp(min=1e-12)
            px = torch.floor(J.fx * a[:, 0] / az + J.cx + 0.5).clamp(-9, J.width + 9).long()
            py = torch.floor(J.fy * a[:, 1] / az + J.cy + 0.5).clamp(-9, J.height + 9).long()
            ok = (a[:, 2] > 0) & (px >= 0) & (px < J.width) & (py >= 0) & (py < J.height)
            flat = torch.where(ok, py * J.width + px, torch.zeros_like(px))
            zj = depth[j].to(torch.float64).reshape(-1)[flat]
            ok &= (zj > 0) & torch.isfinite(zj)
            b = torch.stack([zj * (px.double() - J.cx) / J.fx, zj * (py.double() - J.cy) / J.fy, zj], 1) * u
            e += torch.where(ok, ((a - b) ** 2).sum(1), torch.zeros_like(e)) / (SIGMA_M ** 2 * k1)
        yield {"valid": int(valid.sum()), "idx": idx + off, "world": world, "r": torch.stack(r, 1), "e": e, "c": c,
               "rgb": images[2][i].reshape(-1, 3)[idx].to(torch.float64), "n": cam.width * cam.height}
        off += cam.width * cam.height


def _exact_cloud(case, rig, images):
    got = list(_exact_points(case, rig, images))
    cat = {k: torch.cat([g[k] for g in got]) for k in ("idx", "world", "r", "e", "c", "rgb")}
    valid, n_px = sum(g["valid"] for g in got), rig.n_pixels
    n_gated, bbox = len(cat["idx"]), torch.cat([cat["world"].amin(0), cat["world"].amax(0)])
    top = cat["r"] * 2.0 ** MAX_LEVEL
    inside = ((top >= -BIAS) & (top < BIAS)).all(1)
    cat = {k: v[inside] for k, v in cat.items()}

    def pack(level, k):
        k = k.long() + BIAS
        return (level << 60) | (k[:, 0] << 40) | (k[:, 1] << 20) | k[:, 2]

    zero = torch.zeros(len(cat["idx"]), dtype=torch.int64, device="cuda")
    _, back, dens = torch.unique(pack(zero, torch.floor(cat["r"])), return_inverse=True, return_counts=True)
    level = torch.zeros_like(dens)
    for lv in range(1, MAX_LEVEL + 1):
        level = torch.where(dens >= N_MIN * 4 ** lv, torch.full_like(level, lv), level)
    n_coarse, lv = len(dens), level[back]
    key = pack(lv, torch.floor(cat["r"] * torch.pow(2.0, lv.double())[:, None]))
    keys, cell, count = torch.unique(key, return_inverse=True, return_counts=True)
    order = torch.argsort(cat["idx"], stable=True)
    order = order[torch.argsort(cat["c"][order], descending=True, stable=True)]
    order = order[torch.argsort(cell[order], stable=True)]
    first = torch.cumsum(count, 0) - count
    if case["top_k"]:
        rank = torch.arange(len(order), device="cuda") - first[cell[order]]
        member = order[rank < case["top_k"]]
    else:
        member = order
    rep = cat["idx"][order[first]]
    m = cell[member]
    low = torch.full((len(keys),), math.inf, dtype=torch.float64, device="cuda")
    low.scatter_reduce_(0, m, cat["e"][member], "amin")
    w = cat["c"][member] * torch.exp(low[m] - cat["e"][member])
    total = torch.zeros_like(low).index_add_(0, m, w)
    mean = [torch.zeros(len(keys), 3, dtype=torch.float64, device="cuda").index_add_(0, m, w[:, None] * cat[k][member])
            / total[:, None] for k in ("world", "rgb")]
    cap = max(65536, n_px // 8)
    place = torch.argsort(rep)

    def full(v):
        out = torch.zeros((cap,) + tuple(v.shape[1:]), dtype=v.dtype, device="cuda")
        out[:len(place)] = v[place]
        return out

    out = {"pos": full(mean[0]), "rgb": full(mean[1]), "weight": full(total * torch.exp(-low)),
           "count": full(count.to(torch.int32)), "rep": full(rep.to(torch.int32)), "key": full(keys)}
    n_out = n_gated - int(inside.sum())
    return out, (valid, n_gated, n_out, len(keys), n_coarse), bbox


def exact(case, seed):
    rig, kind = _rig(case), case["kind"]
    frames = [_images(case, rig, seed * 64 + f) for f in range(case["frames"])]
    if kind in ("frame", "graph", "batch"):
        outs = []
        for images in frames:
            out, n, bbox = _exact_cloud(case, rig, images)
            out["pixels_and_cells"] = torch.tensor(n[:4])
            out["extent"] = bbox
            out["error_and_coarse"] = torch.tensor([0, n[4]], dtype=torch.int32)
            outs.append(out)
        return outs
    if kind == "host":
        out, n, bbox = _exact_cloud(case, rig, frames[0])
        return {"status": 0, "cells": n[3], "gated": n[1], "coarse": n[4], "extent": bbox, **out}
    if kind == "points":
        n_px, dev = rig.n_pixels, torch.device("cuda")
        pos = torch.full((n_px, 3), math.nan, dtype=torch.float64, device=dev)
        weight = torch.zeros(n_px, dtype=torch.float64, device=dev)
        for g in _exact_points(case, rig, frames[0]):
            pos[g["idx"]] = g["world"]
            weight[g["idx"]] = g["c"] * torch.exp(-g["e"])
        return {"pos": pos, "weight": weight, "rgb": torch.cat([v.reshape(-1, 3) for v in frames[0][2]])}
    if kind == "screen":
        return [d.to(s.dtype).view(torch.int16) if s.dtype == torch.uint16 else d
                for d, s in zip(_exact_screen(rig, frames[0][0]), frames[0][0])]
    if kind == "confidence":
        return [_exact_confidence(d, rig.depth_scale) for d in frames[0][0]]
    return _exact_mc(rig, frames[0][0], _points(case, rig, frames[0], seed))


def _exact_confidence(d, unit):
    z = d.to(torch.float64) * unit
    ok = (z > 0) & torch.isfinite(z)
    h, w = z.shape
    pz, po = torch.nn.functional.pad(z, (1, 1, 1, 1)), torch.nn.functional.pad(ok, (1, 1, 1, 1))

    def at(dy, dx):
        return pz[1 + dy:1 + dy + h, 1 + dx:1 + dx + w], po[1 + dy:1 + dy + h, 1 + dx:1 + dx + w]

    g2 = torch.zeros_like(z)
    for dy, dx in ((0, 1), (1, 0)):
        (zp, vp), (zm, vm) = at(dy, dx), at(-dy, -dx)
        g = torch.where(vp & vm, (zp - zm) / 2, torch.where(vp, zp - z, torch.where(vm, z - zm, torch.zeros_like(z))))
        g2 += g * g
    n = sum(at(dy, dx)[1].double() for dy in (-1, 0, 1) for dx in (-1, 0, 1)).clamp(min=1)
    near = [(zz - z, vv) for zz, vv in (at(dy, dx) for dy in (-1, 0, 1) for dx in (-1, 0, 1))]
    mean = sum(torch.where(v, e, torch.zeros_like(e)) for e, v in near) / n
    var = sum(torch.where(v, (e - mean) ** 2, torch.zeros_like(e)) for e, v in near) / n
    return torch.where(ok, (0.5 / (1 + 0.5 * g2.sqrt()) + 1.0 / (1 + var)) / 1.5, torch.zeros_like(z))


def _exact_mc(rig, depth, pts):
    p, u = pts.to(torch.float64), rig.depth_scale
    total, seen = torch.zeros(len(p), dtype=torch.float64, device=p.device), torch.zeros_like(p[:, 0], dtype=torch.int32)
    for cam, d in zip(rig.cameras, depth):
        a = p @ torch.as_tensor(cam.R, device=p.device).T + torch.as_tensor(cam.t, device=p.device)
        az = a[:, 2].clamp(min=1e-12)
        x = torch.floor(cam.fx * a[:, 0] / az + cam.cx + 0.5).clamp(-9, cam.width + 9).long()
        y = torch.floor(cam.fy * a[:, 1] / az + cam.cy + 0.5).clamp(-9, cam.height + 9).long()
        ok = (a[:, 2] > 0) & (x >= 0) & (x < cam.width) & (y >= 0) & (y < cam.height)
        z = d.to(torch.float64).reshape(-1)[torch.where(ok, y * cam.width + x, torch.zeros_like(x))] * u
        ok &= (z > 0) & torch.isfinite(z) & (a[:, 2] <= z + F.MC_OCCLUSION_M)
        total += torch.where(ok, (a[:, 2] - z).abs(), torch.zeros_like(z))
        seen += ok.to(torch.int32)
    err = total / seen
    fine = seen > 0
    return {"mc": float(err[fine].mean()), "used": None, "err": None, "seen": None}   # pixels picked in float32
