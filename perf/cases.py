"""Performance cases: the calls that a renderer built on this library makes, from a thumbnail to a 4K frame of
a finely tessellated surface, each through the public entry points of `paper_1811_03510_gb300.ccs`.

A case is a dict of plain values.  `kind` names the call:

  camera   ccs_intersect on the pinhole rays of one image (coherent primary rays)
  bounce   ccs_intersect on the compacted diffuse or mirror rays that leave an image's hits (a small sphere
           beside the large one, as in `shadow`, so that some of them arrive somewhere)
  shadow   ccs_occluded on the compacted shadow rays of an image's hits (any hit, bounded intervals)
  host     ccs_intersect_host_batches: one frame's primary and diffuse rays in page-locked host memory
  frame    ccs_batch_launch: new control points, refit and closest hit of several scenes, one graph replay
  learned  ccs_intersect_learned with a proposal network trained beforehand
  grad     ccs_proposal_grad on one mini-batch of traces
  infer    ccs_proposal_infer on many feature rows

Scenes are the repository's displaced cube-spheres (`n` quads per cube face: 24 n^2 patches, 24 of them
Gregory), seen from `dist` in a direction that the seed gives.  `local` takes the sub-domain boxes in the
patches' own frames.  `engine` is "pairs" (the options a tuned program passes) or "default" (no options).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1811_03510_gb300 import ccs, scenegen

DEV = "cuda"
INF = float("inf")


def listed():
    return [
        # a thumbnail or a picking query on the smallest scene: launches and latency are all there is
        dict(name="thumbnail", kind="camera", n=2, amp=0.0, octaves=3, w=64, h=64, dist=3.0, local=True,
             engine="pairs", depth=8),
        # the first generation of a full-HD frame, as a renderer with tuned options traces it
        dict(name="primary_1080p", kind="camera", n=8, amp=0.05, octaves=3, w=1920, h=1080, dist=3.0, local=True,
             engine="pairs", depth=8),
        # the diffuse generation of that frame: incoherent rays, most of them leave the surface for good
        dict(name="diffuse_1080p", kind="bounce", bounce="diffuse", rays=330000, n=8, amp=0.05, octaves=3, w=1920,
             h=1080, dist=3.0, local=True, engine="pairs", depth=8),
        # first use: a scene and a launch with nothing chosen, on an image of odd sides
        dict(name="defaults_odd", kind="camera", n=8, amp=0.05, octaves=3, w=1283, h=717, dist=3.0, local=False,
             engine="default", depth=8),
        # a 4K frame of a finely tessellated surface: patches of a few pixels, scene data beyond L1
        dict(name="primary_4k_fine", kind="camera", n=64, amp=0.1, octaves=5, w=3840, h=2160, dist=3.0, local=True,
             engine="pairs", depth=8),
        # mirror reflections off that surface: secondary rays with real hits and long BVH walks
        dict(name="mirror_fine", kind="bounce", bounce="mirror", rays=1200000, n=64, amp=0.1, octaves=5, w=2560,
             h=1440, dist=2.2, local=True, engine="pairs", depth=8),
        # next-event estimation: one shadow ray per hit toward a point light, past an occluder
        dict(name="shadow_1080p", kind="shadow", rays=300000, n=8, amp=0.05, octaves=3, w=1920, h=1080, dist=3.0,
             local=True, engine="pairs", depth=8),
        # a host application without device buffers: both generations through the staged pipeline
        dict(name="host_1080p", kind="host", rays=330000, n=8, amp=0.05, octaves=3, w=1920, h=1080, dist=3.0,
             local=True, engine="pairs", depth=8),
        # an animation of several objects of uneven size: repack, refit and trace, one graph replay a frame
        dict(name="animated_frame", kind="frame", scenes=8, n_min=4, n_max=32, rays=70000, amp=0.0, octaves=3, w=512,
             h=512, dist=3.0, local=True, engine="pairs", depth=8),
        # the learned search order on an image, with a trained network
        dict(name="learned_720p", kind="learned", n=8, amp=0.05, octaves=3, w=1280, h=720, dist=3.0, local=True,
             engine="default", depth=8),
        # a training step's gradient at the training batch size
        dict(name="grad_8192", kind="grad", rows=8192),
        # scoring of a held-out trace set
        dict(name="infer_450k", kind="infer", rows=450000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["camera", "camera", "camera", "bounce", "bounce", "shadow", "host", "frame", "learned", "grad",
                       "infer"])
    if kind == "grad":
        return dict(kind=kind, rows=_log(rng, 200, 20000))
    if kind == "infer":
        return dict(kind=kind, rows=_log(rng, 1000, 900000))
    w = _log(rng, 48, 1920)
    c = dict(kind=kind, n=_log(rng, 2, 40), amp=round(rng.uniform(0.0, 0.1), 4), octaves=rng.choice([3, 5]), w=w,
             h=max(16, int(w * rng.uniform(0.5, 1.0))), dist=round(rng.uniform(2.0, 4.0), 3),
             local=rng.random() < 0.7, engine="pairs" if rng.random() < 0.7 else "default",
             depth=rng.choice([6, 7, 8, 8, 8, 9, 10]))
    if rng.random() < 0.5:   # the widths of real images; the others are odd or ragged
        c["w"] = max(64, w // 32 * 32)
    if kind == "bounce":
        c["bounce"] = rng.choice(["diffuse", "mirror"])
    if kind == "frame":
        del c["n"]
        c.update(scenes=rng.randint(2, 10), n_min=rng.randint(2, 6), n_max=rng.randint(8, 28), w=min(c["w"], 512),
                 h=min(c["h"], 512))
    if kind in ("bounce", "shadow", "host", "frame"):   # at most the rays that a full sphere's hits give
        c["rays"] = max(64, int(c["w"] * c["h"] * rng.uniform(0.05, 0.3)))
    if kind == "learned":
        c.update(engine="default", w=min(c["w"], 1280), h=min(c["h"], 720))
    return c


# ------------------------------------------------------------------------------------------- inputs

class _State:
    """What a user's program holds: the scene, the rays, the result buffers and the options."""

    batch = 0
    prop = 0

    def __del__(self):
        if self.batch:
            ccs.ccs_batch_destroy(self.batch)
        if self.prop:
            ccs.ccs_proposal_destroy(self.prop)


def _opts(case, width=0):
    if case["engine"] == "default":
        return None if case["depth"] == 8 else ccs.make_opts(leaf_depth=case["depth"])
    return ccs.make_opts(leaf_depth=case["depth"], pairs=True, image_width=width, cache_slots=1)


def _geometry(case, seed, n=None):
    return scenegen.make_scene(case["n"] if n is None else n, case["amp"], case["octaves"], 1 + seed % 100003)


def _scene(case, P, types):
    return ccs.Scene(P, types, local=case["local"], bvh_width=4 if case["engine"] == "pairs" else 2)


def _unit(v):
    return v / np.linalg.norm(v)


def _eye(case, seed):
    return case["dist"] * _unit(np.random.default_rng(seed + 77).normal(size=3))


def _camera(case, seed):
    """Pinhole rays of a w x h image (60 degrees high) looking at the origin: eight device planes."""
    w, h, eye = case["w"], case["h"], _eye(case, seed)
    fwd = _unit(-eye)
    right = _unit(np.cross(fwd, [0.0, 0.0, 1.0] if abs(fwd[2]) < 0.9 else [1.0, 0.0, 0.0]))
    up = np.cross(right, fwd)
    th = math.tan(math.radians(30.0))
    x = ((torch.arange(w, device=DEV, dtype=torch.float64) + 0.5) * (2.0 / w) - 1.0) * (th * w / h)
    y = (1.0 - (torch.arange(h, device=DEV, dtype=torch.float64) + 0.5) * (2.0 / h)) * th
    x, y = x[None, :].expand(h, w).reshape(-1), y[:, None].expand(h, w).reshape(-1)
    d = [fwd[k] + right[k] * x + up[k] * y for k in range(3)]
    s = torch.rsqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2])
    o = [torch.full((w * h,), float(eye[k]), device=DEV) for k in range(3)]
    return o + [(q * s).float().contiguous() for q in d] + \
        [torch.zeros(w * h, device=DEV), torch.full((w * h,), INF, device=DEV)]


def _bounce(case, seed, sc, cam, kind, light=None):
    """The compacted secondary rays that leave the hits of the camera rays: the case's number of them, the
    image's rays over again where it has fewer."""
    hits = ccs.intersect(sc, cam, ccs.make_opts(leaf_depth=case["depth"], pairs=True))
    if kind == "diffuse":
        r = ccs.gen_diffuse(sc, cam, hits, seed=1 + seed, leaf_depth=case["depth"])
    elif kind == "mirror":
        r = ccs.gen_mirror(sc, cam, hits, leaf_depth=case["depth"])
    else:
        r = ccs.gen_shadow(sc, cam, hits, light, leaf_depth=case["depth"])
    keep = (r[7] >= r[6]).nonzero().squeeze(1)
    keep = keep[torch.arange(case["rays"], device=DEV) % keep.numel()]
    return [q.index_select(0, keep).contiguous() for q in r]


def _occluded_geometry(case, seed):
    """The sphere, a small sphere between it and a light beside the camera, and that light."""
    g = _geometry(case, seed)
    eye = _eye(case, seed)
    light = 1.4 * eye + 1.2 * _unit(np.cross(eye, [0.3, 0.5, 0.8]))
    small = scenegen.make_scene(2, 0.0, name="occluder")
    P = np.concatenate([g.P, (0.35 * small.P + 0.5 * light).astype(np.float32)])
    return P, np.concatenate([g.types, small.types]), [float(q) for q in light]


def _features(rows, seed):
    """Feature rows as the traversal makes them: points and lengths in patch units, unit vectors, a flag."""
    gen = torch.Generator(device=DEV).manual_seed(seed + 11)
    f = torch.randn(rows, 24, device=DEV, generator=gen) * 0.6
    for a in (3, 18):
        f[:, a:a + 3] /= f[:, a:a + 3].norm(dim=1, keepdim=True).clamp_min(1e-6)
    f[:, 21] = f[:, 21].abs().clamp_max(4.0)
    f[:, 22] = (f[:, 3:6] * f[:, 18:21]).sum(1)
    f[:, 23] = (torch.rand(rows, device=DEV, generator=gen) < 0.06).float()
    return f.contiguous(), torch.randint(0, 64, (rows,), device=DEV, generator=gen).to(torch.uint8)


def _params(seed):
    """FP32 network parameters: He-normal weights, small biases."""
    r = np.random.default_rng(seed + 5)
    parts = []
    for fan, out in ((24, 64), (64, 64), (64, 64)):
        parts += [r.normal(size=out * fan) * math.sqrt(2.0 / fan), r.normal(size=out) * 0.05]
    return np.concatenate(parts).astype(np.float32)


def _trained(sc, cam, depth):
    """A proposal fitted to the traces of the image: a short training of the kind a program does once."""
    n, cap = int(cam[0].numel()), 1 << 19
    feat, lab = torch.zeros(cap, 24, device=DEV), torch.zeros(cap, dtype=torch.uint8, device=DEV)
    cnt = torch.zeros(1, dtype=torch.int32, device=DEV)
    hits = ccs.alloc_hits(n)
    ccs.ccs_trace_export(sc.handle, cam, n, hits, ccs.make_opts(leaf_depth=depth), feat, lab, cap, cnt)
    m = min(int(cnt.item()), cap)
    prop = ccs.ccs_proposal_create(seed=1)
    rows = min(4096, m)
    if rows:
        pick = torch.randperm(m, device=DEV, generator=torch.Generator(device=DEV).manual_seed(1))
        feat, lab = feat[pick].contiguous(), lab[pick].contiguous()
        for k in range(64):
            a = (k * rows) % (m - rows + 1)
            ccs.ccs_proposal_train_step(prop, feat[a:], lab[a:], rows, 2e-3)
    torch.cuda.synchronize()
    return prop


def _pinned(planes):
    """The planes as rows of one page-locked host block."""
    block = torch.empty(len(planes), planes[0].numel(), dtype=torch.float32).pin_memory()
    for row, q in zip(block, planes):
        row.copy_(q)
    return block


def prepare(case, seed):
    s = _State()
    s.case, kind = case, case["kind"]
    if kind in ("grad", "infer"):
        s.feat, s.lab = _features(case["rows"], seed)
        s.prop = ccs.ccs_proposal_create(seed=1)
        ccs.ccs_proposal_set_params(s.prop, _params(seed))
        s.grad, s.loss = torch.empty(9920, device=DEV), torch.empty(1, device=DEV)
        s.logits = torch.empty(case["rows"], 64, device=DEV)
        s.cells = torch.empty(case["rows"], dtype=torch.uint8, device=DEV)
        s.pmax = torch.empty(case["rows"], device=DEV)
        return s
    cam = _camera(case, seed)
    if kind == "frame":
        sizes = np.linspace(case["n_min"], case["n_max"], case["scenes"]).round().astype(int)
        rng = np.random.default_rng(seed)
        s.scenes, s.points, s.rays, s.hits = [], [], [], []
        for k, n in enumerate(sizes):
            g = _geometry(case, seed + k, int(n))
            sc = _scene(case, g.P, g.types)
            rest = torch.from_numpy(g.P).to(DEV)
            wave, phase = (torch.from_numpy(rng.uniform(2.0, 6.0, 3).astype(np.float32)).to(DEV) for _ in range(2))
            Q = rest + 0.02 * torch.sin(wave * rest + phase)
            s.points.append([Q[..., c].contiguous().reshape(-1) for c in range(3)])
            d = _bounce(case, seed + k, sc, cam, "diffuse")
            s.scenes.append(sc)
            s.rays.append([torch.cat([a, b]).contiguous() for a, b in zip(cam, d)])
            s.hits.append(ccs.alloc_hits(int(s.rays[-1][0].numel())))
        s.batch = ccs.ccs_batch_create(s.scenes, s.rays, s.hits)
        for k, q in enumerate(s.points):
            ccs.ccs_batch_set_points(s.batch, k, *q)
        ccs.ccs_batch_capture(s.batch, ccs.CCS_BATCH_UPDATE | ccs.CCS_BATCH_REFIT | ccs.CCS_BATCH_INTERSECT,
                              _opts(case))
        return s
    if kind in ("bounce", "shadow"):
        P, types, light = _occluded_geometry(case, seed)
        s.scene = _scene(case, P, types)
        s.rays = _bounce(case, seed, s.scene, cam, case.get("bounce", "shadow"), light)
        s.n, s.opts, s.rs = case["rays"], _opts(case), ccs.rays_struct(s.rays)
        s.out = torch.empty(s.n, dtype=torch.uint8, device=DEV)
        s.hits = ccs.alloc_hits(s.n)
        s.hs = ccs.hits_struct(s.hits)
        return s
    g = _geometry(case, seed)
    s.scene = _scene(case, g.P, g.types)
    s.opts = _opts(case, case["w"])
    s.rays = cam
    if kind == "host":
        s.blocks = [_pinned(cam), _pinned(_bounce(case, seed, s.scene, cam, "diffuse"))]
        s.count = [int(b.shape[1]) for b in s.blocks]
        s.outs = [torch.empty(4, m, dtype=torch.float32).pin_memory() for m in s.count]
        s.rs = [ccs.rays_struct(list(b)) for b in s.blocks]
        s.hs = [ccs.hits_struct(list(b)) for b in s.outs]
        s.opts = [s.opts, _opts(case)]
        return s
    if kind == "learned":
        s.prop = _trained(s.scene, cam, case["depth"])
        s.opts = ccs.make_opts(leaf_depth=case["depth"])
    s.n = int(s.rays[0].numel())
    s.hits = ccs.alloc_hits(s.n)
    s.rs, s.hs = ccs.rays_struct(s.rays), ccs.hits_struct(s.hits)
    return s


def run(s):
    kind = s.case["kind"]
    if kind in ("camera", "bounce"):
        if s.opts is None:
            return ccs.intersect(s.scene, s.rays)
        ccs.ccs_intersect(s.scene.handle, s.rs, s.n, s.hs, s.opts)
        return s.hits
    if kind == "shadow":
        ccs.ccs_occluded(s.scene.handle, s.rs, s.n, s.out, s.opts)
        return s.out
    if kind == "host":
        ccs.ccs_intersect_host_batches(s.scene.handle, s.rs, s.count, s.hs, s.opts)
        return [[b[0], b[1], b[2], b[3].view(torch.int32)] for b in s.outs]
    if kind == "frame":
        ccs.ccs_batch_launch(s.batch)
        return s.hits
    if kind == "learned":
        ccs.ccs_intersect_learned(s.scene.handle, s.prop, s.rs, s.n, s.hs, s.opts, 0.0)
        return s.hits
    if kind == "grad":
        ccs.ccs_proposal_grad(s.prop, s.feat, s.lab, s.case["rows"], s.grad, s.loss)
        return {"grad": s.grad, "loss": s.loss}
    ccs.ccs_proposal_infer(s.prop, s.feat, s.case["rows"], s.logits, s.cells, s.pmax)
    return {"logits": s.logits, "cells": s.cells, "pmax": s.pmax}


# ------------------------------------------------------------------------- what a pass cannot do without

def _covered(case):
    """Share of the image that the unit sphere covers."""
    r = math.tan(math.asin(min(0.99, 1.0 / case["dist"]))) / math.tan(math.radians(30.0))   # of half the height
    return min(1.0, math.pi * r * r / 4.0 * case["h"] / case["w"])


def work(case):
    """Bytes: rays in, hits out, the scene's points once.  Operations: a few BVH nodes per ray (34 each), and for
    a ray that hits, one split (360) per level of the subdivision (the counts this method needs on these
    scenes); the network's products."""
    if case["kind"] in ("grad", "infer"):
        rows, mults = case["rows"], 24 * 64 + 2 * 64 * 64
        if case["kind"] == "grad":
            return {"bytes": rows * (24 * 4 + 1) + 2 * 9920 * 4, "flops": rows * (6 * mults - 2 * 24 * 64)}
        return {"bytes": rows * (24 * 4 + 64 * 4 + 1 + 4) + 9920 * 4, "flops": rows * 2 * mults}
    px, hit, steps = case["w"] * case["h"], _covered(case), 2 * case["depth"] * 360
    if case["kind"] == "frame":
        sizes = np.linspace(case["n_min"], case["n_max"], case["scenes"]).round()
        points = float((24 * sizes * sizes).sum()) * 240
        second = case["rays"] * (2 * 360 + 13 * 34)
        return {"bytes": (px + case["rays"]) * case["scenes"] * 48 + points,
                "flops": case["scenes"] * (px * (hit * steps + 5 * 34) + second)}
    scene = 24 * case["n"] ** 2 * 240
    primary = {"bytes": px * 48 + scene, "flops": px * (hit * steps + 5 * 34)}
    if case["kind"] in ("camera", "learned"):
        return primary
    second = {"bytes": case["rays"] * 48 + scene, "flops": case["rays"] * (2 * 360 + 13 * 34)}
    if case["kind"] == "bounce":
        return second
    if case["kind"] == "shadow":
        return {"bytes": case["rays"] * 33 + scene, "flops": second["flops"]}
    return {k: primary[k] + second[k] for k in primary}


# --------------------------------------------------------------------------------- the same in 64 bits

def _crop(a, b):
    """Matrix [.., 4, 4] that maps the control points of a cubic to those of its restriction to [a, b]."""
    rows = []
    for t in ((a, a, a), (a, a, b), (a, b, b), (b, b, b)):
        x, y, z = t
        rows.append(torch.stack([(1 - x) * (1 - y) * (1 - z),
                                 x * (1 - y) * (1 - z) + y * (1 - x) * (1 - z) + z * (1 - x) * (1 - y),
                                 x * y * (1 - z) + x * z * (1 - y) + y * z * (1 - x), x * y * z], -1))
    return torch.stack(rows, -2)


def _peak(a, b, at):
    """Maximum over [a, b] of 3 t (1-t)^2 (at = 1/3) or 3 t^2 (1-t) (at = 2/3)."""
    t = torch.minimum(torch.maximum(torch.full_like(a, at), a), b)
    return 3 * t * (1 - t) * (1 - t) if at < 0.5 else 3 * t * t * (1 - t)


def _ratio(a, b):
    return torch.where(a + b == 0, 0.5, a / (a + b).clamp_min(1e-300))


def _node(pts, greg, u0, u1, v0, v1):
    """Lower control grid [m, j, i, 3] of the node and the displacement [m, 3] of its upper bound: the patch
    itself cropped (Bezier), or the bound over the extreme inner points (Gregory), cropped."""
    p = pts[:, :16].clone()
    d = torch.zeros(len(pts), 3, dtype=pts.dtype, device=pts.device)
    lo = [(u0, v1), (1 - u0, v0), (u1, 1 - v1), (1 - u1, 1 - v0)]
    hi = [(u1, v0), (1 - u1, v1), (u0, 1 - v0), (1 - u0, 1 - v1)]
    bu, bv = [_peak(u0, u1, q) for q in (1 / 3, 2 / 3)], [_peak(v0, v1, q) for q in (1 / 3, 2 / 3)]
    for m, slot in enumerate((5, 6, 9, 10)):
        pu, pv = pts[:, slot], pts[:, 16 + m]
        a, b = (pv + _ratio(*q)[:, None] * (pu - pv) for q in (lo[m], hi[m]))
        p[:, slot] = torch.where(greg[:, None], torch.minimum(a, b), pu)
        d += torch.where(greg[:, None], (bu[m & 1] * bv[m >> 1])[:, None] * (a - b).abs(), 0.0)
    return torch.einsum("mjp,mpqc,miq->mjic", _crop(v0, v1), p.reshape(-1, 4, 4, 3), _crop(u0, u1)), d


def _slab(lo, hi, o, inv, c0, c1):
    a, b = (lo - o) * inv, (hi - o) * inv
    return torch.maximum(torch.minimum(a, b).amax(1), c0), torch.minimum(torch.maximum(a, b).amin(1), c1)


def _frames(P):
    """Rows of each patch's own frame (z along the corner quad's normal, x along its u edge)."""
    a, b, e = P[:, 15] - P[:, 0], P[:, 12] - P[:, 3], P[:, 3] - P[:, 0]
    z = torch.linalg.cross(a, b)
    z = z / z.norm(dim=1, keepdim=True)
    x = e - (e * z).sum(1, keepdim=True) * z
    x = x / x.norm(dim=1, keepdim=True)
    return torch.stack([x, torch.linalg.cross(z, x), z], 1).float().double()


def _exact_hits(case, seed):
    """Closest leaf (t, u, v) of every camera ray: all nodes that a ray enters, level by level."""
    g = _geometry(case, seed)
    P = torch.from_numpy(g.P).to(DEV).double()
    greg = torch.from_numpy(g.types).to(DEV) != 0
    rays = [q.double() for q in _camera(case, seed)]
    o, d = torch.stack(rays[:3], 1), torch.stack(rays[3:6], 1)
    lo, hi = torch.where(greg[:, None], P.amin(1), P[:, :16].amin(1)), torch.where(greg[:, None], P.amax(1), P[:, :16].amax(1))
    mid = ((lo.float() + hi.float()) * 0.5).double()
    R = _frames(P) if case["local"] else torch.eye(3, dtype=P.dtype, device=DEV).expand(len(P), 3, 3)
    Q = torch.einsum("pkc,psc->psk", R, P - mid[:, None])
    found = []
    for a in range(0, len(o), 16384):
        oo, inv = o[a:a + 16384], 1.0 / d[a:a + 16384]
        near, far = torch.full((len(oo), len(P)), 0.0, dtype=P.dtype, device=DEV), torch.full((len(oo), len(P)), INF, dtype=P.dtype, device=DEV)
        for k in range(3):
            x, y = (lo[None, :, k] - oo[:, None, k]) * inv[:, None, k], (hi[None, :, k] - oo[:, None, k]) * inv[:, None, k]
            near, far = torch.maximum(near, torch.minimum(x, y)), torch.minimum(far, torch.maximum(x, y))
        r, p = (near <= far).nonzero(as_tuple=True)
        found.append((r + a, p, near[r, p], far[r, p]))
    ray, pid, c0, c1 = (torch.cat(q) for q in zip(*found))
    o3 = o[ray] - mid[pid]
    po, pinv = torch.einsum("mkc,mc->mk", R[pid], o3), 1.0 / torch.einsum("mkc,mc->mk", R[pid], d[ray])
    tau = 2.0 ** -19 * (1 + o3.abs().sum(1)) if case["local"] else torch.zeros_like(c0)
    cu, cv = torch.zeros_like(c0), torch.zeros_like(c0)
    for level in range(2 * case["depth"]):
        su, sv = 2.0 ** -((level + 1) // 2), 2.0 ** -(level // 2)
        grid, up = _node(Q[pid], greg[pid], cu * su, (cu + 1) * su, cv * sv, (cv + 1) * sv)
        axis, half, kept = 2 - level % 2, torch.full((1,), 0.5, dtype=P.dtype, device=DEV), []
        for side in (0, 1):
            m = _crop(half * side, half * (side + 1))[0]
            child = torch.einsum("ai,mjic->mjac", m, grid) if axis == 2 else torch.einsum("aj,mjic->maic", m, grid)
            b0, b1 = child.amin((1, 2)), child.amax((1, 2)) + up
            e = ((tau[:, None] - (b1 - b0)) * 0.5).clamp_min(0.0)
            t0, t1 = _slab(b0 - e, b1 + e, po, pinv, c0, c1)
            ok = (t0 <= t1).nonzero().squeeze(1)
            nu, nv = (cu * 2 + side, cv) if axis == 2 else (cu, cv * 2 + side)
            kept.append([q[ok] for q in (ray, pid, t0, t1, po, pinv, tau, nu, nv)])
        ray, pid, c0, c1, po, pinv, tau, cu, cv = (torch.cat(q) for q in zip(*kept))
    order = torch.argsort(pid * 4.0 ** case["depth"] + cv * 2.0 ** case["depth"] + cu, stable=True)
    order = order[torch.argsort(c0[order], stable=True)]
    order = order[torch.argsort(ray[order], stable=True)]
    first = torch.ones(len(order), dtype=torch.bool, device=DEV)
    first[1:] = ray[order][1:] != ray[order][:-1]
    w = order[first]
    t, u, v = torch.full((len(o),), INF, dtype=P.dtype, device=DEV), torch.zeros(len(o), dtype=P.dtype, device=DEV), torch.zeros(len(o), dtype=P.dtype, device=DEV)
    t[ray[w]], u[ray[w]], v[ray[w]] = c0[w], (cu[w] + 0.5) * 2.0 ** -case["depth"], (cv[w] + 0.5) * 2.0 ** -case["depth"]
    return [t, u, v, None]


def _exact_net(case, seed):
    feat, lab = _features(case["rows"], seed)
    flat = torch.from_numpy(_params(seed)).to(DEV)
    infer = case["kind"] == "infer"
    round16 = (lambda q: q.float().bfloat16().double()) if infer else (lambda q: q)   # the stored inputs of inference
    parts, at = [], 0
    for fan in (24, 64, 64):
        for shape in ((64, fan), (64,)):
            m = math.prod(shape)
            q = flat[at:at + m].reshape(shape).double()
            parts.append((round16(q) if len(shape) == 2 else q).requires_grad_(not infer))
            at += m
    x = feat.double()
    for k in range(3):
        z = round16(x) @ parts[2 * k].T + parts[2 * k + 1]
        x = torch.relu(z) if k < 2 else z
    if infer:
        return {"logits": x, "cells": None, "pmax": torch.softmax(x, 1).amax(1)}
    loss = torch.nn.functional.cross_entropy(x, lab.long())
    loss.backward()
    return {"grad": torch.cat([q.grad.reshape(-1) for q in parts]), "loss": loss.detach().reshape(1)}


def exact(case, seed):
    if case["kind"] in ("grad", "infer"):
        return _exact_net(case, seed)
    # hits pick one of many leaves: in 64 bits only where all nodes of all rays can be listed in a few seconds
    if case["kind"] in ("camera", "learned") and case["w"] * case["h"] * 24 * case["n"] ** 2 <= 4e9:
        return _exact_hits(case, seed)
    return None
