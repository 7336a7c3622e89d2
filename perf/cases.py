"""Performance cases of the LDNI framework: the calls its users make, each with
the inputs such a call meets, over the range of sizes it is used at.

A case names a `kind` (one public call or the pair of calls of a frame) and its
sizes.  Meshes are generated on the GPU from the seed; operands that a case
takes as given (the images of a Boolean, a chain, an offset, a contour) are
sampled here with plain torch, so that they do not depend on the sampler that
other cases measure.  `exact` restates the paper's definitions in 64 bits; the
steps that are decisions by definition (the snap to the 8-bit subpixel grid,
the order of FP32 depths, the sphere test of an offset) are taken in FP32 with
single roundings, as defined.

Results have one size for all seeds of a case: kept buffers are sized by the
case with room to spare (zero beyond the samples), and where a call allocates
its results to size, another seed moves the same solid by whole pixels, which
changes every ray but not the number of samples.
"""
import ctypes
import math

import numpy as np
import torch

import paper_1009_0794_gb300 as ldni
from paper_1009_0794_gb300 import _lib, autograd, capacity

WIDTH = 1.0  # the cube [-W/2, W/2]^3 (calls that allocate their results: see _width)


# ---- the cases -------------------------------------------------------------------

def listed():
    return [
        # A user's first call: a 1,280-triangle solid at preview resolution, buffers allocated and sized
        # by the call itself (the smallest work: launches and the one readback).
        dict(name="sample_call_1k_64", kind="sample", api="call", shape="sphere", noise="uniform", tris=1280, res=64,
             packed=False),
        # The paper's own setting: a model of half a million triangles at 512^2, with 8-bit normals.
        dict(name="sample_packed_523k_512", kind="sample", api="call", shape="flower", noise="none", tris=523264,
             res=512, packed=True),
        # Repeated exact sampling of a scanned model at the finest resolution in use, buffers kept.
        dict(name="sample_plan_1m3_2048", kind="sample", api="plan", shape="sphere", noise="octave", tris=1310720,
             res=2048, packed=False),
        # One frame of the interactive modeller: a deforming model sampled in one pass, united with a resident
        # tool, the volumes of the result returned (the benchmark's step).
        dict(name="frame_1m3_1024", kind="frame", tris=1310720, knot=16384, res=1024),
        # A subtraction of two resident multi-layer solids with thin pieces removed, at an odd resolution.
        dict(name="boolean_diff_777", kind="boolean", api="many", op="diff", a="flower", b="knot", res=777, eps=1e-5),
        # One small Boolean as an interactive edit makes it: one image, scratch allocated, the size read back.
        dict(name="boolean_call_128", kind="boolean", api="call", op="union", a="sphere", b="torus", res=128, eps=0.0),
        # A library of parts sampled in one call: uneven meshes and resolutions, some with deep rays.
        dict(name="batch_48", kind="batch", count=48, tris_lo=1000, tris_hi=200000, res_hi=512),
        # A sweep: 64 placements of a 20,000-triangle part united in order.
        dict(name="chain_64x20k_512", kind="chain", parts=64, tris=20000, res=512),
        # Shape optimisation: the volume of a 200,000-triangle solid and its gradient.
        dict(name="gradient_200k_512", kind="gradient", tris=200000, res=512),
        # Inside status of all grid nodes, the first step of meshing a result.
        dict(name="nodes_1024", kind="nodes", res=1024),
        # Cell vertices of a united solid for meshing, at a usual export resolution.
        dict(name="contour_256", kind="contour", res=256),
        # Offsetting as in the paper's examples: 128^2 images grown by 2.5 pixels.
        dict(name="offset_128_r2.5", kind="offset", res=128, radius=2.5, inner=False),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["sample", "sample", "frame", "boolean", "boolean", "batch", "chain", "gradient", "nodes",
                       "contour", "offset"])
    if kind == "sample":
        shape = rng.choice(["sphere", "flower", "torus", "knot", "box"])
        return dict(kind=kind, api=rng.choice(["call", "plan"]), shape=shape,
                    noise=rng.choice(["none", "octave", "uniform"]) if shape == "sphere" else "none",
                    tris=12 if shape == "box" else _log_int(rng, 1000, 1200000), res=_log_int(rng, 32, 1900),
                    packed=rng.random() < 0.3)
    if kind == "frame":
        return dict(kind=kind, tris=_log_int(rng, 10000, 1300000), knot=_log_int(rng, 4096, 65536),
                    res=_log_int(rng, 128, 1280))
    if kind == "boolean":
        return dict(kind=kind, api=rng.choice(["call", "many", "many"]), op=rng.choice(["union", "inter", "diff"]),
                    a=rng.choice(["sphere", "flower", "knot"]), b=rng.choice(["torus", "knot"]),
                    res=_log_int(rng, 40, 1400), eps=rng.choice([0.0, 1e-5]))
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(4, 48), tris_lo=1000, tris_hi=_log_int(rng, 5000, 200000),
                    res_hi=rng.choice([64, 128, 256, 512]))
    if kind == "chain":
        return dict(kind=kind, parts=rng.randint(3, 64), tris=_log_int(rng, 1000, 20000), res=_log_int(rng, 64, 640))
    if kind == "gradient":
        return dict(kind=kind, tris=_log_int(rng, 2000, 400000), res=_log_int(rng, 64, 900))
    if kind == "nodes":
        return dict(kind=kind, res=_log_int(rng, 40, 1100))
    if kind == "contour":
        return dict(kind=kind, res=_log_int(rng, 30, 320))
    return dict(kind=kind, res=_log_int(rng, 30, 140), radius=round(rng.uniform(0.8, 2.6), 2),
                inner=rng.random() < 0.4)


# ---- meshes ----------------------------------------------------------------------

def _rand(seed, *shape):
    g = torch.Generator(device="cuda").manual_seed(int(seed) & 0x7FFFFFFFFFFF)
    return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64)


def _finish(v, t):
    """FP32 vertices (multiples of 2^-22, so that moves by whole pixels of a
    power-of-two pitch are exact) and int32 triangles, turned outward."""
    a, b, c = v[t[:, 0]], v[t[:, 1]], v[t[:, 2]]
    if float((a * torch.linalg.cross(b, c)).sum()) < 0:
        t = t[:, [0, 2, 1]]
    return (torch.round(v * 2.0 ** 22) * 2.0 ** -22).to(torch.float32).contiguous(), t.to(torch.int32).contiguous()


def _moved(mesh, seed, res, width):
    """The mesh moved by up to a sixteenth of the cube in whole pixels, its
    triangles listed from another one on."""
    u = [float(x) for x in _rand(seed, 4).cpu()]
    h = width / res
    shift = [(round((2 * x - 1) * res / 16)) * h for x in u[:3]]
    v = (mesh[0].to(torch.float64) + torch.tensor(shift, dtype=torch.float64, device="cuda")).to(torch.float32)
    return v, torch.roll(mesh[1], int(u[3] * mesh[1].shape[0]), 0).contiguous()


def _width(case):
    """The cube of a sampling call that allocates its results: its pitch is a
    power of two (_moved)."""
    if case["kind"] == "sample" and case["api"] == "call":
        return case["res"] * 2.0 ** -math.ceil(math.log2(case["res"]))
    return WIDTH


def _sample_mesh(case, seed):
    if case["api"] == "plan":
        return _mesh(case["shape"], case["tris"], seed, case["noise"])
    v, t = _mesh(case["shape"], case["tris"], 5, case["noise"])
    w = _width(case)
    return _moved((torch.round(v * (0.85 * w) * 2.0 ** 22) * 2.0 ** -22, t), seed, case["res"], w)


def _quads(nu, nv):
    """Triangles of a periodic nu x nv quad grid, vertex (i, j) -> i nv + j."""
    i = torch.arange(nu, device="cuda")[:, None]
    j = torch.arange(nv, device="cuda")[None, :]
    a, b = i * nv + j, (i + 1) % nu * nv + j
    c, d = (i + 1) % nu * nv + (j + 1) % nv, i * nv + (j + 1) % nv
    return torch.stack([a, b, c, a, c, d], -1).reshape(-1, 3)


def _sphere(tris, r, noise, amp, seed, centre=(0.0, 0.0, 0.0)):
    """Cube sphere (12 n^2 triangles) with smooth ("octave") or per-vertex
    ("uniform") radial noise; vertices numbered in order of first use."""
    n = max(2, int(round((tris / 12.0) ** 0.5)))
    a, b = torch.meshgrid(torch.arange(n + 1, device="cuda"), torch.arange(n + 1, device="cuda"), indexing="ij")
    pts, faces = [], []
    q = torch.arange(n, device="cuda")
    p00 = (q[:, None] * (n + 1) + q[None, :]).reshape(-1)
    quad = torch.stack([p00, p00 + n + 1, p00 + n + 2, p00, p00 + n + 2, p00 + 1], -1).reshape(-1, 3)
    for axis in range(3):
        for side in (0, n):
            p = torch.empty(n + 1, n + 1, 3, dtype=torch.int64, device="cuda")
            p[..., axis], p[..., (axis + 1) % 3], p[..., (axis + 2) % 3] = side, a, b
            faces.append((quad if side else quad[:, [0, 2, 1]]) + len(pts) * (n + 1) ** 2)
            pts.append(p.reshape(-1, 3))
    pts, faces = torch.cat(pts), torch.cat(faces)
    key = (pts[:, 0] * (n + 1) + pts[:, 1]) * (n + 1) + pts[:, 2]
    uniq, inv = torch.unique(key, return_inverse=True)
    use = inv[faces].reshape(-1)
    first = torch.full_like(uniq, use.numel()).scatter_reduce_(0, use, torch.arange(use.numel(), device="cuda"), "amin")
    order = torch.argsort(first)
    rank = torch.empty_like(order)
    rank[order] = torch.arange(order.numel(), device="cuda")
    lat = torch.stack([uniq // (n + 1) ** 2, uniq // (n + 1) % (n + 1), uniq % (n + 1)], -1)[order]
    d = torch.tan((lat.to(torch.float64) * (2.0 / n) - 1.0) * (math.pi / 4))
    d = d / d.norm(dim=1, keepdim=True)
    rad = torch.full((d.shape[0],), r, dtype=torch.float64, device="cuda")
    if noise == "octave" and amp > 0:
        u = _rand(seed, 24, 4)
        f = torch.zeros_like(rad)
        for k in range(24):
            kv = u[k, :3] * 2 - 1
            kv = kv / kv.norm() * (2.0 * 2.0 ** (k // 6))
            f += 0.5 ** (k // 6) * torch.sin(d @ kv + 2 * math.pi * u[k, 3])
        rad = rad + f * (amp / f.abs().max())
    elif noise == "uniform" and amp > 0:
        rad = rad + (_rand(seed, d.shape[0]) * 2 - 1) * min(amp, 0.6 * r / n)
    return _finish(d * rad[:, None] + torch.tensor(centre, dtype=torch.float64, device="cuda"), rank[inv[faces]])


def _angles(n, phase=0.0):
    return (torch.arange(n, device="cuda", dtype=torch.float64) + phase) * (2 * math.pi / n)


def _torus(tris, R, r, seed, noise=0.0, centre=(0.0, 0.0, 0.0), ratio=2):
    """Quad torus about z with about `tris` triangles; per-vertex tube noise."""
    nv = max(4, int(round((tris / (2.0 * ratio)) ** 0.5)))
    nu = max(4, int(round(tris / 2.0 / nv)))
    u, w = _angles(nu, float(_rand(seed, 1)))[:, None], _angles(nv, 0.25)[None, :]
    rr = torch.full((nu, nv), r, dtype=torch.float64, device="cuda")
    if noise > 0:
        rr = rr + (_rand(seed + 1, nu, nv) * 2 - 1) * noise
    x, y, z = (R + rr * torch.cos(w)) * torch.cos(u), (R + rr * torch.cos(w)) * torch.sin(u), rr * torch.sin(w)
    v = torch.stack([x, y, z], -1).reshape(-1, 3) + torch.tensor(centre, dtype=torch.float64, device="cuda")
    return _finish(v, _quads(nu, nv))


def _flower(tris, seed):
    """Star-shaped flower r = 0.3 + 0.08 cos(8 phi) sin^2(theta)."""
    n = max(8, int(round((tris / 2.0) ** 0.5)))
    th = (math.pi / n) * torch.arange(1, n, device="cuda", dtype=torch.float64)[:, None]
    ph = _angles(n)[None, :]
    turn = float(_rand(seed, 1)) * 2 * math.pi
    rad = 0.3 + 0.08 * torch.cos(8 * ph + turn) * torch.sin(th) ** 2
    v = torch.stack([rad * torch.sin(th) * torch.cos(ph), rad * torch.sin(th) * torch.sin(ph), rad * torch.cos(th)], -1)
    poles = torch.tensor([[0.0, 0.0, 0.3], [0.0, 0.0, -0.3]], dtype=torch.float64, device="cuda")
    j = torch.arange(n, device="cuda")
    jn, top, last = (j + 1) % n, (n - 1) * n, (n - 2) * n
    a = (torch.arange(n - 2, device="cuda")[:, None] * n + j).reshape(-1)
    an = (torch.arange(n - 2, device="cuda")[:, None] * n + jn).reshape(-1)
    t = torch.cat([torch.stack([torch.full_like(j, top), j, jn], -1),
                   torch.stack([a, a + n, an + n, a, an + n, an], -1).reshape(-1, 3),
                   torch.stack([torch.full_like(j, top + 1), last + jn, last + j], -1)])
    return _finish(torch.cat([v.reshape(-1, 3), poles]), t)


def _knot(tris, seed, tube=0.035):
    """Tube around the (2, 3) torus knot."""
    side = max(6, int(round((tris / 16.0) ** 0.5)))
    ring = max(24, int(round(tris / 2.0 / side)))
    t = _angles(ring, float(_rand(seed, 1)))
    c, s, one = torch.cos, torch.sin, torch.zeros_like(t)
    er, ep = torch.stack([c(2 * t), s(2 * t), one], -1), torch.stack([-s(2 * t), c(2 * t), one], -1)
    ez = torch.tensor([0.0, 0.0, 1.0], dtype=torch.float64, device="cuda")
    rad = (0.25 + 0.1 * c(3 * t))[:, None]
    p = rad * er + 0.1 * s(3 * t)[:, None] * ez
    tan = -0.3 * s(3 * t)[:, None] * er + 2 * rad * ep + 0.3 * c(3 * t)[:, None] * ez
    tan = tan / tan.norm(dim=1, keepdim=True)
    nrm = c(3 * t)[:, None] * er + s(3 * t)[:, None] * ez
    nrm = nrm - (nrm * tan).sum(1, keepdim=True) * tan
    nrm = nrm / nrm.norm(dim=1, keepdim=True)
    bi = torch.linalg.cross(tan, nrm)
    w = _angles(side)[None, :, None]
    return _finish((p[:, None] + tube * (c(w) * nrm[:, None] + s(w) * bi[:, None])).reshape(-1, 3), _quads(ring, side))


def _box(seed):
    lo, hi = -0.45 + 0.1 * _rand(seed, 3), 0.45 - 0.1 * _rand(seed + 1, 3)
    v = torch.stack([torch.stack([(hi if (k >> a) & 1 else lo)[a] for a in range(3)]) for k in range(8)])
    t = torch.tensor([[0, 2, 3], [0, 3, 1], [4, 5, 7], [4, 7, 6], [0, 1, 5], [0, 5, 4], [2, 6, 7], [2, 7, 3],
                      [0, 4, 6], [0, 6, 2], [1, 3, 7], [1, 7, 5]], device="cuda")
    return _finish(v, t)


def _mesh(shape, tris, seed, noise="octave"):
    if shape == "sphere":
        at = [0.02 * float(x) for x in _rand(seed + 9, 3).cpu()]
        return _sphere(tris, 0.35, noise, 0.03 if noise == "uniform" else 0.05, seed, at)
    if shape == "torus":
        return _torus(tris, 0.25, 0.1, seed, centre=(0.12, 0.0, 0.02))
    if shape == "flower":
        return _flower(tris, seed)
    if shape == "knot":
        return _knot(tris, seed)
    return _box(seed)


def _batch_meshes(case, seed):
    """Noisy spheres and tori, sizes in log-uniform steps."""
    out = []
    for m in range(case["count"]):
        f = (m * 0.6180339887) % 1.0
        tris = int(case["tris_lo"] * (case["tris_hi"] / case["tris_lo"]) ** f)
        res = max(64, case["res_hi"] >> ((m * 5 + 3) % 4))
        u = [float(x) for x in _rand(77 + m, 2).cpu()]
        if m % 2:
            r = 0.2 + 0.2 * u[0]
            mesh = _sphere(tris, r, "octave", 0.1 * r, 300 + m)
        else:
            rr = 0.05 + 0.1 * u[1]
            mesh = _torus(tris, 0.2 + 0.08 * u[0], rr, 300 + m, noise=0.2 * rr, ratio=4)
        out.append(_moved(mesh, seed + 1000 * m, res, WIDTH) + (res,))
    return out


# ---- the definitions in plain torch ----------------------------------------------

def _crossings(v, t, res, axis, width=WIDTH):
    """Every crossing of one image, in CSR order: offsets, FP64 depth, FP64
    normal, triangle, ray (Definitions 1-4; top-left rule on the snapped
    triangle)."""
    scale = torch.tensor(np.float32(res * 256.0 / width), device="cuda")
    q = torch.round((v + width / 2) * scale).to(torch.int64)
    t = t.to(torch.int64)
    u, w = (axis + 1) % 3, (axis + 2) % 3
    qu, qw, a = q[:, u][t], q[:, w][t], v[:, axis].to(torch.float64)[t]
    lo = lambda x: ((x.amin(1) + 127) >> 8).clamp_min(0)  # noqa: E731
    hi = lambda x: ((x.amax(1) - 128) >> 8).clamp_max(res - 1)  # noqa: E731
    i0, i1, j0, j1 = lo(qu), hi(qu), lo(qw), hi(qw)
    area = (qu[:, 1] - qu[:, 0]) * (qw[:, 2] - qw[:, 0]) - (qw[:, 1] - qw[:, 0]) * (qu[:, 2] - qu[:, 0])
    tri = torch.nonzero((i0 <= i1) & (j0 <= j1) & (area != 0)).reshape(-1)
    flip = (area[tri] < 0)[:, None]
    ccw = lambda x: torch.where(flip, x[tri][:, [0, 2, 1]], x[tri])  # noqa: E731
    qu, qw, a, area = ccw(qu), ccw(qw), ccw(a), area[tri].abs()
    wd, npx = (i1 - i0 + 1)[tri], ((i1 - i0 + 1) * (j1 - j0 + 1))[tri]
    i0, j0 = i0[tri], j0[tri]
    ends = npx.cumsum(0)
    step = 1 << 25  # pairs handled at a time
    rows = []
    at = 0
    while at < tri.numel():
        base = int(ends[at - 1]) if at else 0
        to = max(at + 1, int(torch.searchsorted(ends, base + step)))
        sel = torch.arange(at, min(to, tri.numel()), device="cuda")
        k = sel.repeat_interleave(npx[sel])
        x = torch.arange(k.numel(), device="cuda") + base - (ends - npx)[k]
        i, j = i0[k] + x % wd[k], j0[k] + x // wd[k]
        cu, cw = 256 * i + 128, 256 * j + 128
        e, ok = [], None
        for p, n in ((0, 1), (1, 2), (2, 0)):
            du, dw = (qu[:, n] - qu[:, p])[k], (qw[:, n] - qw[:, p])[k]
            f = du * (cw - qw[k, p]) - dw * (cu - qu[k, p])
            own = (f > 0) | ((f == 0) & ((dw > 0) | ((dw == 0) & (du < 0))))
            ok = own if ok is None else ok & own
            e.append(f)
        hit = torch.nonzero(ok).reshape(-1)
        k, A = k[hit], area[k[hit]].to(torch.float64)
        lam = [e[m][hit].to(torch.float64) / A for m in (1, 2, 0)]  # the edge opposite vertex m
        rows.append((j[hit] * res + i[hit], tri[k], sum(lam[m] * a[k, m] for m in range(3))))
        at = to
    if not rows:
        rows = [(torch.zeros(0, dtype=torch.int64, device="cuda"),) * 2 + (torch.zeros(0, dtype=torch.float64,
                                                                                        device="cuda"),)]
    ray, tri, d = (torch.cat(x) for x in zip(*rows))
    order = torch.sort(d.to(torch.float32), stable=True).indices  # triangles already ascend
    order = order[torch.sort(ray[order], stable=True).indices]
    ray, tri, d = ray[order], tri[order], d[order]
    offsets = torch.zeros(res * res + 1, dtype=torch.int64, device="cuda")
    offsets[1:] = torch.bincount(ray, minlength=res * res).cumsum(0)
    p = v.to(torch.float64)[t[tri]]
    n = torch.linalg.cross(p[:, 1] - p[:, 0], p[:, 2] - p[:, 0])
    return dict(offsets=offsets, depth=d, n=n / n.norm(dim=1, keepdim=True), tri=tri, ray=ray)


def _images(mesh, res, axes=(0, 1, 2), width=WIDTH):
    return [_crossings(mesh[0], mesh[1], res, a, width) for a in axes]


def _rounded(img):
    """The image as an FP32 framework holds it."""
    return dict(img, depth=img["depth"].to(torch.float32), n=img["n"].to(torch.float32))


def _ldni(img, grid, axis):
    n = img["n"].to(torch.float32)
    return ldni.LDNI(grid, axis, img["offsets"].to(torch.int32), img["depth"].to(torch.float32).contiguous(),
                     n[:, 0].contiguous(), n[:, 1].contiguous(), n[:, 2].contiguous(), img["tri"].to(torch.int32),
                     img["depth"].numel())


def _drop_thin(rows, key, eps):
    """Boundaries come in entering / leaving pairs: those thinner than eps go."""
    d = key.to(torch.float32)
    keep = ~((d[rows[1::2]] - d[rows[0::2]]) < eps)
    return rows[keep.repeat_interleave(2)]


def _merge(A, B, op, eps, res):
    """A op B by inside-counters (Section 4.1), FP32 depths ordering."""
    ray = torch.cat([A["ray"], B["ray"]])
    depth = torch.cat([A["depth"], B["depth"]])
    n, tri = torch.cat([A["n"], -B["n"] if op == "diff" else B["n"]]), torch.cat([A["tri"], B["tri"] | (1 << 31)])
    from_b = torch.cat([torch.zeros_like(A["ray"]), torch.ones_like(B["ray"])])
    order = torch.sort(depth.to(torch.float32), stable=True).indices
    order = order[torch.sort(ray[order], stable=True).indices]
    d, r, fb = depth[order].to(torch.float32), ray[order], from_b[order]
    new = torch.ones_like(r, dtype=torch.bool)
    new[1:] = (r[1:] != r[:-1]) | (d[1:] != d[:-1])
    group = new.cumsum(0) - 1
    ng = int(group[-1]) + 1 if group.numel() else 0
    ca = torch.zeros(ng, dtype=torch.int64, device="cuda").index_add_(0, group, 1 - fb)
    cb = torch.zeros(ng, dtype=torch.int64, device="cuda").index_add_(0, group, fb)
    sa, sb = (ca.cumsum(0) & 1).bool(), (cb.cumsum(0) & 1).bool()  # every ray closes, so states reset by themselves
    now = {"union": sa | sb, "inter": sa & sb, "diff": sa & ~sb}[op]
    was = torch.cat([now[:1] & False, now[:-1]])
    start = torch.nonzero(new).reshape(-1)
    src = torch.where((ca & 1).bool(), start, start + ca)[now != was]  # A's samples come first in a group
    src = _drop_thin(src, d, eps)
    src = order[src]
    counts = torch.bincount(ray[src], minlength=res * res)
    offsets = torch.zeros(res * res + 1, dtype=torch.int64, device="cuda")
    offsets[1:] = counts.cumsum(0)
    return dict(offsets=offsets, depth=depth[src], n=n[src], tri=tri[src], ray=ray[src])


def _volume(img, res):
    return (img["depth"][1::2] - img["depth"][0::2]).to(torch.float64).sum() * (WIDTH / res) ** 2


def _node(t, res):
    """Node coordinates: fl32(o + fl32((t + 1/2) h))."""
    h = torch.tensor(np.float32(WIDTH) / np.float32(res), device="cuda")
    return (t.to(torch.float32) + 0.5) * h + (-WIDTH / 2)


def _inside(imgs, res):
    """Inside status [i, j, k] of the grid nodes: 2-of-3 vote of the images."""
    votes = torch.zeros(res, res, res, dtype=torch.uint8, device="cuda")
    for a, img in enumerate(imgs):
        c = _node(torch.arange(res, device="cuda"), res)
        t = torch.searchsorted(c, img["depth"].to(torch.float32).contiguous(), right=True)  # first node above d
        flips = torch.zeros(res * res, res + 1, dtype=torch.uint8, device="cuda")
        flips.view(-1).index_add_(0, img["ray"] * (res + 1) + t, torch.ones_like(t, dtype=torch.uint8))
        bits = (flips[:, :res].cumsum(1, dtype=torch.uint8) & 1).view(res, res, res)  # [v, u, along]
        votes += bits.permute(*((2, 1, 0), (0, 2, 1), (1, 0, 2))[a])
    return votes >= 2


# ---- preparing and running -------------------------------------------------------

def _outputs(L):
    d = {"offsets": L.offsets, "depth": L.depth, "tri": L.tri}
    if L.packed:
        d["nrm8"] = L.nrm8
    else:
        d.update(nx=L.nx, ny=L.ny, nz=L.nz)
    return d


def _exact_outputs(img, packed=False, cap=0):
    pad = lambda x: torch.cat([x.to(torch.float64), x.new_zeros(max(0, cap - x.numel()), dtype=torch.float64)])  # noqa: E731
    d = {"offsets": img["offsets"], "depth": pad(img["depth"]), "tri": None}
    if packed:
        d["nrm8"] = None
    else:
        d.update((k, pad(img["n"][:, a])) for a, k in enumerate(("nx", "ny", "nz")))
    return d


def _grid(res, width=WIDTH):
    return ldni.Grid.cube((-width / 2,) * 3, width, res)


def _cleared(images):
    for L in images:
        for x in _outputs(L).values():
            x.zero_()
    return images


def _boolean_operands(case, seed):
    axes = (0,) if case["api"] == "call" else (0, 1, 2)
    A = _images(_mesh(case["a"], 200000, seed), case["res"], axes)
    B = _images(_mesh(case["b"], 16384, seed + 1), case["res"], axes)
    return axes, [_rounded(x) for x in A], [_rounded(x) for x in B]


def _room(case):
    """Samples an image of the case's result has room for."""
    res = case["res"]
    est = lambda shape: int(0.6 * _samples(shape, res)) + 64 * res  # noqa: E731
    if case["kind"] == "sample":
        return est(case["shape"])
    if case["kind"] == "frame":
        return est("sphere") + est("knot")
    if case["kind"] == "boolean":
        return est(case["a"]) + est(case["b"])
    if case["kind"] == "chain":
        return int(0.11 * case["parts"] * res * res) + 64 * res
    return int(3 * math.pi * (0.38 + case["radius"] / res) ** 2 * res * res) + 64 * res  # an offset


def _united(case, seed):
    """The united solid (noisy sphere and knot) of the meshing cases, FP32."""
    res = case["res"]
    A, B = _images(_mesh("sphere", 50000, seed), res), _images(_mesh("knot", 16384, seed + 1), res)
    return [_merge(_rounded(a), _rounded(b), "union", 0.0, res) for a, b in zip(A, B)]


def _chain_parts(case, seed):
    """One part swept along a helix: translated meshes."""
    v, t = _torus(case["tris"], 0.1, 0.04, seed, ratio=1)
    turns = 1.0 + float(_rand(seed + 1, 1))
    out = []
    for k in range(case["parts"]):
        s = k / max(1, case["parts"] - 1)
        ang = 2 * math.pi * turns * s
        shift = torch.tensor([0.15 * math.cos(ang), 0.15 * math.sin(ang), 0.4 * (s - 0.5)], dtype=torch.float64,
                             device="cuda")
        out.append(((v.to(torch.float64) + shift).to(torch.float32), t))
    return out


def _trained_net():
    """A small capacity network, trained as the framework trains its own."""
    meshes = [_sphere(20 * f * f, 0.3, "octave", a, f) for f, a in ((24, 0.02), (48, 0.05), (64, 0.0), (96, 0.07))]
    X, label = capacity.build_dataset(meshes, 512)
    net = capacity.CapacityNet(seed=0)
    net.fit(X, label, steps=300, batch=512)
    return net


def prepare(case, seed):
    kind, res, s = case["kind"], case.get("res"), {"case": case}
    if kind == "batch":
        _prepare_batch(s, _batch_meshes(case, seed))
        return s
    g = s["grid"] = _grid(res, _width(case))
    if kind == "sample":
        v, t = s["mesh"] = _sample_mesh(case, seed)
        if case["api"] == "plan":
            s["plan"] = ldni.SamplePlan(v.shape[0], t.shape[0], g, [_room(case)] * 3, packed=case["packed"])
            _cleared(s["plan"].outs)
    elif kind == "frame":
        v, t = s["mesh"] = _mesh("sphere", case["tris"], seed)
        s["net"] = _trained_net()
        s["plan"] = ldni.LearnedPlan(v.shape[0], t.shape[0], g, [_room(case)] * 3, 24 * res * res, net=s["net"])
        _cleared(s["plan"].outs)
        knot = _images(_mesh("knot", case["knot"], seed + 1), res)
        s["tool"] = [_ldni(x, g, a) for a, x in enumerate(knot)]
        _boolean_buffers(s, (0, 1, 2))
    elif kind == "boolean":
        axes, A, B = _boolean_operands(case, seed)
        s["A"], s["B"] = ([_ldni(x, g, a) for a, x in zip(axes, X)] for X in (A, B))
        _boolean_buffers(s, axes)
    elif kind == "chain":
        meshes = _chain_parts(case, seed)
        images = [[_ldni(_crossings(v, t, res, a), g, a) for v, t in meshes] for a in range(3)]
        s["chain"], s["finish"] = ldni.union_chain_many(images, capacities=[_room(case)] * 3)
        s["parts"] = images
        s["chain"]()
        _cleared(s["finish"]())
    elif kind == "gradient":
        v, t = _sphere(case["tris"], 0.35, "octave", 0.03, seed)
        s["verts"], s["tris"] = v.requires_grad_(True), t
    elif kind in ("nodes", "contour"):
        s["images"] = [_ldni(x, g, a) for a, x in enumerate(_united(case, seed))]
        s["ws"] = _workspace("ldni_classify_nodes_workspace_size", res)
        s["inside"] = torch.empty(res, res, (res + 31) // 32, dtype=torch.int32, device="cuda")
        s["info"] = ldni.new_info()
        if kind == "contour":
            s["bound"] = min((res - 1) ** 3, int(4 * _samples("sphere", res)) + 6 * (res - 1) ** 2 + 64)
            s["cells"] = torch.zeros(6 * res * res, ldni.CELL_DTYPE.itemsize, dtype=torch.uint8, device="cuda")
            s["cws"] = _workspace("ldni_contour_workspace_size", res, s["bound"])
            s["layers"] = (_lib.Layers * 3)(*[L.c() for L in s["images"]])
    elif kind == "offset":
        H = s["images"] = [_ldni(x, g, a) for a, x in enumerate(_images(_mesh("flower", 60000, seed), res))]
        s["radius"] = case["radius"] * WIDTH / res
        s["outs"] = _cleared([ldni.empty_layers(g, a, _room(case)) for a in range(3)])
        s["n"] = (ctypes.c_int64 * 3)(*[L.n for L in H])
        s["ws"] = torch.empty(ldni.offset_workspace_size([L.n for L in H], res, s["radius"], WIDTH), dtype=torch.uint8,
                              device="cuda")
        s["info"] = ldni.new_info()
        s["H"], s["out"] = ((_lib.Layers * 3)(*[L.c() for L in X]) for X in (H, s["outs"]))
    return s


def _workspace(query, *sizes):
    sz = ctypes.c_size_t(0)
    _lib.check(getattr(_lib.load(), query)(*sizes, ctypes.byref(sz)), query)
    return torch.empty(sz.value, dtype=torch.uint8, device="cuda")


def _boolean_buffers(s, axes):
    count = len(axes)
    s["outs"] = _cleared([ldni.empty_layers(s["grid"], a, _room(s["case"])) for a in axes])
    s["ws"] = torch.empty(ldni.boolean_many_workspace_size(s["grid"].res, count), dtype=torch.uint8, device="cuda")
    s["infos"] = torch.zeros(count, _lib.INFO_BYTES // 8, dtype=torch.int64, device="cuda")
    s["vols"] = torch.zeros(count, dtype=torch.float64, device="cuda")


def _prepare_batch(s, meshes):
    """A batch through the C ABI, every image of every mesh carved from one
    array per field, so that the results are six tensors."""
    count = len(meshes)
    sized = [[L.n for L in ldni.sample(v, t, _grid(res), "all")] for v, t, res in meshes]
    pad = lambda k: (k + 63) // 64 * 64  # noqa: E731
    rows = sum(3 * pad(res * res + 1) for _, _, res in meshes)
    total = max(64, sum(pad(n) for ns in sized for n in ns))
    out = {k: torch.zeros(rows if k == "offsets" else total, device="cuda",
                          dtype=torch.int32 if k in ("offsets", "tri") else torch.float32)
           for k in ("offsets", "depth", "nx", "ny", "nz", "tri")}
    items = (_lib.BatchItem * count)()
    r = k = 0
    for m, (v, t, res) in enumerate(meshes):
        it, g = items[m], _grid(res)
        it.verts, it.tris, it.nv, it.nt, it.grid = v.data_ptr(), t.data_ptr(), v.shape[0], t.shape[0], g.c()
        for a in range(3):
            n, N = sized[m][a], res * res + 1
            L = ldni.LDNI(g, a, out["offsets"][r:r + N], *(out[f][k:k + n] for f in ("depth", "nx", "ny", "nz", "tri")), n)
            it.out[a] = L.c()
            r, k = r + pad(N), k + pad(n)
    s.update(meshes=meshes, out=out, items=items, count=count)
    s["items_dev"] = torch.frombuffer(bytearray(bytes(memoryview(items))), dtype=torch.uint8).cuda()
    s["ws"] = _workspace("ldni_sample_batch_workspace_size", ctypes.byref(items), count)
    s["infos"] = torch.zeros(count, _lib.INFO_BYTES // 8, dtype=torch.int64, device="cuda")


def run(state):
    s, case = state, state["case"]
    kind = case["kind"]
    if kind == "sample":
        if case["api"] == "plan":
            s["plan"].run(*s["mesh"])
            outs = s["plan"].outs
        else:
            outs = ldni.sample(*s["mesh"], s["grid"], "all", packed=case["packed"])
        return [_outputs(L) for L in outs]
    if kind == "frame":
        s["plan"].run(*s["mesh"])
        U = ldni.boolean_many(s["plan"].outs, s["tool"], "union", outs=s["outs"], ws=s["ws"], infos=s["infos"],
                              sync=False, vols=s["vols"])
        return {"model": [_outputs(L) for L in s["plan"].outs], "union": [_outputs(L) for L in U], "volumes": s["vols"]}
    if kind == "boolean":
        if case["api"] == "call":
            return _outputs(ldni.boolean(s["A"][0], s["B"][0], case["op"], case["eps"], out=s["outs"][0]))
        U = ldni.boolean_many(s["A"], s["B"], case["op"], case["eps"], outs=s["outs"], ws=s["ws"], infos=s["infos"],
                              sync=False, vols=s["vols"])
        return {"result": [_outputs(L) for L in U], "volumes": s["vols"]}
    if kind == "batch":
        _lib.check(_lib.load().ldni_sample_batch(s["items_dev"].data_ptr(), ctypes.byref(s["items"]), s["count"],
                                                 s["infos"].data_ptr(), s["ws"].data_ptr(), s["ws"].numel(),
                                                 _stream()), "ldni_sample_batch")
        return s["out"]
    if kind == "chain":
        s["chain"]()
        return [_outputs(L) for L in s["finish"]()]
    if kind == "gradient":
        vol = autograd.LDNIVolume.apply(s["verts"], s["tris"], s["grid"], "all")
        return {"volume": vol, "grad": torch.autograd.grad(vol, s["verts"])[0]}
    if kind in ("nodes", "contour"):
        inside = ldni.classify_nodes(s["images"], out=s["inside"], ws=s["ws"], info=s["info"], sync=False)
        if kind == "nodes":
            return inside
        cells = s["cells"]
        _lib.check(_lib.load().ldni_contour_cells(s["layers"], ctypes.byref(s["grid"].c()), inside.data_ptr(),
                                                  s["bound"], cells.data_ptr(), cells.shape[0], s["info"].data_ptr(),
                                                  s["cws"].data_ptr(), s["cws"].numel(), _stream()),
                   "ldni_contour_cells")
        return {"cell": cells.view(torch.int64)[:, 0], "labels, npts, nvert": cells.view(torch.int32)[:, 2:5],
                "v": cells.view(torch.float32)[:, 6:]}
    _lib.check(_lib.load().ldni_offset(s["H"], s["n"], ctypes.byref(s["grid"].c()), s["radius"], int(case["inner"]), 0.0,
                                       s["out"], s["info"].data_ptr(), s["ws"].data_ptr(), s["ws"].numel(),
                                       _stream()), "ldni_offset")
    return [_outputs(L) for L in s["outs"]]


def _stream():
    return ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)


# ---- exact results ---------------------------------------------------------------

def exact(case, seed):
    kind, res = case["kind"], case.get("res")
    if kind == "sample":
        imgs = _images(_sample_mesh(case, seed), res, width=_width(case))
        return [_exact_outputs(x, case["packed"], _room(case) if case["api"] == "plan" else 0) for x in imgs]
    if kind == "frame":
        imgs = _images(_mesh("sphere", case["tris"], seed), res)
        knot = [_rounded(x) for x in _images(_mesh("knot", case["knot"], seed + 1), res)]
        U = [_merge(a, dict(b, depth=b["depth"].to(torch.float64), n=b["n"].to(torch.float64)), "union", 0.0, res)
             for a, b in zip(imgs, knot)]
        cap = _room(case)
        return {"model": [_exact_outputs(x, cap=cap) for x in imgs], "union": [_exact_outputs(x, cap=cap) for x in U],
                "volumes": torch.stack([_volume(x, res) for x in U])}
    if kind == "boolean":
        _, A, B = _boolean_operands(case, seed)
        U = [_merge(a, b, case["op"], case["eps"], res) for a, b in zip(A, B)]
        if case["api"] == "call":
            return _exact_outputs(U[0], cap=_room(case))
        U = [dict(x, depth=x["depth"].to(torch.float64)) for x in U]
        return {"result": [_exact_outputs(x, cap=_room(case)) for x in U], "volumes": torch.stack([_volume(x, res) for x in U])}
    if kind == "batch":
        return _exact_batch(_batch_meshes(case, seed))
    if kind == "chain":
        parts = [[_rounded(x) for x in _images(m, res)] for m in _chain_parts(case, seed)]
        out = []
        for a in range(3):
            acc = parts[0][a]
            for p in parts[1:]:
                acc = _merge(acc, p[a], "union", 0.0, res)
            out.append(_exact_outputs(acc, cap=_room(case)))
        return out
    if kind == "gradient":
        return _exact_gradient(_sphere(case["tris"], 0.35, "octave", 0.03, seed), res)
    if kind == "contour":
        return _exact_contour(_united(case, seed), res)
    if kind == "offset":
        H = [_rounded(x) for x in _images(_mesh("flower", 60000, seed), res)]
        return [_exact_outputs(x, cap=_room(case))
                for x in _exact_offset(H, res, case["radius"] * WIDTH / res, case["inner"])]
    return None  # inside bits of the nodes: whole numbers


def _exact_batch(meshes):
    pad = lambda x, k: torch.cat([x, x.new_zeros((-x.numel()) % k)])  # noqa: E731
    out = {k: [] for k in ("offsets", "depth", "nx", "ny", "nz")}
    for v, t, res in meshes:
        for img in _images((v, t), res):
            for k, x in _exact_outputs(img).items():
                if k in out:
                    out[k].append(pad(x, 64))
    return dict({k: torch.cat(x) for k, x in out.items()}, tri=None)


def _exact_gradient(mesh, res):
    """Mean volume of the three images and its gradient with the crossings
    held fixed: d(depth) / d(V_j) = lambda_j n / n_a."""
    v, t = mesh[0].to(torch.float64), mesh[1].to(torch.int64)
    grad, vols, h = torch.zeros_like(v), [], WIDTH / res
    for a in range(3):
        img = _crossings(mesh[0], mesh[1], res, a)
        vols.append(_volume(img, res))
        u, w = (a + 1) % 3, (a + 2) % 3
        ids = t[img["tri"]]
        p = v[ids]
        e1, e2 = p[:, 1] - p[:, 0], p[:, 2] - p[:, 0]
        n = torch.linalg.cross(e1, e2)
        xu = (img["ray"] % res + 0.5) * h - WIDTH / 2 - p[:, 0, u]
        xw = (img["ray"] // res + 0.5) * h - WIDTH / 2 - p[:, 0, w]
        l1 = (xu * e2[:, w] - e2[:, u] * xw) / n[:, a]
        l2 = (e1[:, u] * xw - e1[:, w] * xu) / n[:, a]
        pos = torch.arange(ids.shape[0], device="cuda") - img["offsets"][img["ray"]]
        c = (2.0 * (pos & 1) - 1.0) * h * h / 3.0 / n[:, a]
        for k, lam in enumerate((1 - l1 - l2, l1, l2)):
            grad.index_add_(0, ids[:, k], torch.where((n[:, a] != 0)[:, None], (c * lam)[:, None] * n, 0.0))
    return {"volume": sum(vols) / 3.0, "grad": grad}


def _exact_offset(H, res, r, inner):
    """The solid united with (minus) a sphere about every sample: intervals of
    all spheres per ray, covered by counting; at a change the first source in
    the order H, sphere 0, 1, ... whose own state changes gives the sample."""
    r32 = torch.tensor(np.float32(r), device="cuda")
    r2 = r32 * r32
    C = []
    for a, img in enumerate(H):
        c = torch.empty(img["depth"].numel(), 3, dtype=torch.float32, device="cuda")
        c[:, a], c[:, (a + 1) % 3] = img["depth"], _node(img["ray"] % res, res)
        c[:, (a + 2) % 3] = _node(img["ray"] // res, res)
        C.append(c)
    C = torch.cat(C)
    k = int(math.ceil(r * res / WIDTH)) + 1
    out = []
    for b, img in enumerate(H):
        u, w = (b + 1) % 3, (b + 2) % 3
        iu, iw = (torch.round((C[:, x].to(torch.float64) / WIDTH + 0.5) * res - 0.5).to(torch.int64) for x in (u, w))
        rows = []
        for dj in range(-k, k + 1):
            for di in range(-k, k + 1):
                i, j = iu + di, iw + dj
                du, dw = _node(i, res) - C[:, u], _node(j, res) - C[:, w]
                q = du * du + dw * dw
                s = torch.nonzero((i >= 0) & (j >= 0) & (i < res) & (j < res) & (q < r2)).reshape(-1)
                rows.append((j[s] * res + i[s], s, du[s], dw[s], (r2 - q)[s]))
        ray, sph, du, dw, t2 = (torch.cat(x) for x in zip(*rows))
        t32, t64, cb = t2.sqrt(), t2.to(torch.float64).sqrt(), C[sph, b]
        lo, hi = cb - t32, cb + t32
        met = torch.zeros(res * res, dtype=torch.bool, device="cuda")
        met[ray] = True
        use = torch.nonzero(lo < hi).reshape(-1)
        # events: H's samples, then the spheres' entering and leaving ones
        nh, ns = img["depth"].numel(), use.numel()
        two = torch.cat([use, use])
        e_ray, e_d = torch.cat([img["ray"], ray[two]]), torch.cat([img["depth"], lo[use], hi[use]])
        e_src = torch.cat([torch.full_like(img["ray"], -1), sph[two]])
        e_cov = torch.cat([torch.zeros_like(img["ray"]), torch.ones_like(use), -torch.ones_like(use)])
        order = torch.sort(e_src, stable=True).indices
        order = order[torch.sort(e_d[order], stable=True).indices]
        order = order[torch.sort(e_ray[order], stable=True).indices]
        d, er = e_d[order], e_ray[order]
        new = torch.ones_like(er, dtype=torch.bool)
        new[1:] = (er[1:] != er[:-1]) | (d[1:] != d[:-1])
        start, group = torch.nonzero(new).reshape(-1), new.cumsum(0) - 1
        is_h = (e_src[order] < 0).to(torch.int64)
        zero = torch.zeros(start.numel(), dtype=torch.int64, device="cuda")
        ch, cov = zero.index_add(0, group, is_h), zero.index_add(0, group, e_cov[order])
        sh, sc = (ch.cumsum(0) & 1).bool(), cov.cumsum(0) > 0
        now = (sh & ~sc) if inner else (sh | sc)
        was = torch.cat([now[:1] & False, now[:-1]])
        pick = torch.where((ch & 1).bool(), start, start + ch)  # H first, then the lowest sphere
        src = order[pick[now != was]]
        untouched = torch.nonzero(~met[img["ray"]]).reshape(-1)  # rays no sphere meets keep H as it is
        src = torch.cat([src[met[e_ray[src]]], untouched])
        src = src[torch.sort(e_d[src], stable=True).indices]
        src = src[torch.sort(e_ray[src], stable=True).indices]
        sphere = src >= nh
        at = two[(src - nh).clamp_min(0)]
        sign = torch.where(src - nh >= ns, 1.0, -1.0).to(torch.float64)
        own = src.clamp_max(nh - 1)
        depth, n = img["depth"].to(torch.float64)[own], img["n"].to(torch.float64)[own]
        sn = torch.empty(src.numel(), 3, dtype=torch.float64, device="cuda")
        sn[:, b], sn[:, u], sn[:, w] = sign * t64[at], du[at].to(torch.float64), dw[at].to(torch.float64)
        sn = sn / float(r32) * (-1.0 if inner else 1.0)
        depth = torch.where(sphere, cb[at].to(torch.float64) + sign * t64[at], depth)
        offsets = torch.zeros(res * res + 1, dtype=torch.int64, device="cuda")
        offsets[1:] = torch.bincount(e_ray[src], minlength=res * res).cumsum(0)
        out.append(dict(offsets=offsets, depth=depth, n=torch.where(sphere[:, None], sn, n)))
    return out


def _exact_contour(imgs, res):
    """Cell vertices of Steps 2-3 (Section 5.1): edges typed and regularised,
    outside corners flooded through empty edges, one QEF vertex per cluster."""
    n, inside = res - 1, _inside(imgs, res)  # [i, j, k]
    dev = inside.device
    active = torch.zeros(n, n, n, dtype=torch.bool, device=dev)
    edges = []  # per axis: dense edge index [i, j, k] and the kept samples
    for a, img in enumerate(imgs):
        u, w = (a + 1) % 3, (a + 2) % 3
        c = _node(torch.arange(res, device=dev), res)
        t = torch.searchsorted(c, img["depth"].contiguous(), right=True) - 1
        s = torch.nonzero((t >= 0) & (t < n)).reshape(-1)
        t, ray = t[s], img["ray"][s]
        pos = [None] * 3
        pos[a], pos[u], pos[w] = t, ray % res, ray // res
        flat = (pos[0] * res + pos[1]) * res + pos[2]
        grp_id, grp, cnt = torch.unique_consecutive(flat, return_inverse=True, return_counts=True)
        first = cnt.cumsum(0) - cnt
        lo_in = inside.reshape(-1)[grp_id]
        d, na = img["depth"][s].to(torch.float64), img["n"][s][:, a]
        mid = ((c[t].to(torch.float64) + c[t + 1].to(torch.float64)) / 2)
        dist, fits = (d - mid).abs(), na * torch.where(lo_in[grp], 1.0, -1.0).to(na.dtype) > 0
        best = torch.zeros_like(first)
        score = torch.full(first.shape, math.inf, dtype=torch.float64, device=dev)
        for m in range(int(cnt.max()) if cnt.numel() else 0):
            g = torch.nonzero(cnt > m).reshape(-1)
            at = first[g] + m
            sc = dist[at] + torch.where(fits[at], 0.0, 1e6)
            better = sc < score[g]
            best[g[better]], score[g[better]] = at[better], sc[better]
        index = torch.full((res ** 3,), -1, dtype=torch.int64, device=dev)
        index[grp_id] = torch.arange(grp_id.numel(), device=dev)
        point = torch.empty(s.numel(), 3, dtype=torch.float64, device=dev)
        point[:, a] = d
        point[:, u], point[:, w] = _node(ray % res, res).to(torch.float64), _node(ray // res, res).to(torch.float64)
        edges.append(dict(index=index, cnt=cnt, first=first, best=best, point=point, mid=mid,
                          normal=img["n"][s].to(torch.float64), s=s))
        touched = index.view(res, res, res) >= 0
        step = [0, 0, 0]
        step[a] = 1
        hi = tuple(slice(step[k], res) for k in range(3))
        lo = tuple(slice(0, res - step[k]) for k in range(3))
        touched[lo] |= inside[lo] != inside[hi]
        for x in (0, 1):
            for y in (0, 1):
                off = [0, 0, 0]
                off[u], off[w] = x, y
                active |= touched[tuple(slice(off[k], off[k] + n) for k in range(3))]
    k, j, i = torch.nonzero(active.permute(2, 1, 0)).unbind(1)  # ascending i + n (j + n k)
    at = lambda x, y, z: ((i + x) * res + j + y) * res + k + z  # noqa: E731
    M = i.numel()
    sgn = torch.stack([inside.reshape(-1)[at(c & 1, (c >> 1) & 1, c >> 2)] for c in range(8)], 1)
    info = []  # per cell edge: axis, corners, group (or -1)
    for a in range(3):
        u, w = (a + 1) % 3, (a + 2) % 3
        for x in (0, 1):
            for y in (0, 1):
                off = [0, 0, 0]
                off[u], off[w] = x, y
                q0 = off[0] + 2 * off[1] + 4 * off[2]
                info.append((a, q0, q0 + (1 << a), edges[a]["index"][at(*off)]))
    lab = torch.where(sgn, 99, torch.arange(8, device=dev))
    for _ in range(8):  # the lowest corner of each cluster
        for a, q0, q1, g in info:
            joined = (g < 0) & ~sgn[:, q0] & ~sgn[:, q1]
            low = torch.minimum(lab[:, q0], lab[:, q1])
            lab[:, q0], lab[:, q1] = torch.where(joined, low, lab[:, q0]), torch.where(joined, low, lab[:, q1])
    root = lab == torch.arange(8, device=dev)
    number = root.cumsum(1) - 1
    lab = torch.where(sgn, 15, torch.gather(number, 1, lab.clamp_max(7)))
    ncl = root.sum(1)
    AtA = torch.zeros(M * 4, 3, 3, dtype=torch.float64, device=dev)
    Atb, mass = (torch.zeros(M * 4, 3, dtype=torch.float64, device=dev) for _ in range(2))
    npts, surf = torch.zeros(M * 4, dtype=torch.int64, device=dev), torch.zeros(M, dtype=torch.bool, device=dev)
    cells = torch.arange(M, device=dev)

    def add(mask, label, a, sample):
        q = cells[mask] * 4 + label[mask]
        p, nr = edges[a]["point"][sample[mask]], edges[a]["normal"][sample[mask]]
        AtA.index_add_(0, q, nr[:, :, None] * nr[:, None, :])
        Atb.index_add_(0, q, nr * (nr * p).sum(1, keepdim=True))
        mass.index_add_(0, q, p)
        npts.index_add_(0, q, torch.ones_like(q))

    for a, q0, q1, g in info:
        E, has = edges[a], g >= 0
        gg = g.clamp_min(0)
        if not E["cnt"].numel():
            E = None
        in0, in1 = sgn[:, q0], sgn[:, q1]
        surf |= (in0 != in1) | (has & ~in0 & ~in1)
        if E is None:
            continue
        add(has & (in0 != in1), torch.where(in0, lab[:, q1], lab[:, q0]), a, E["best"][gg])
        both, many = has & ~in0 & ~in1, E["cnt"][gg] >= 2
        s0 = E["first"][gg]
        s1 = s0 + E["cnt"][gg] - 1
        add(both & many, lab[:, q0], a, s0)
        add(both & many, lab[:, q1], a, s1)
        near0 = E["point"][s0, a] < E["mid"][s0]
        add(both & ~many, torch.where(near0, lab[:, q0], lab[:, q1]), a, s0)
    keep = torch.nonzero(surf & (ncl > 0)).reshape(-1)
    v = torch.zeros(M, 4, 3, dtype=torch.float64, device=dev)
    for g in range(4):
        rows = keep[ncl[keep] > g]
        q = rows * 4 + g
        full = npts[q] > 0
        rf, qf = rows[full], q[full]
        if rf.numel():
            m = mass[qf] / npts[qf][:, None]
            lam, V = (x.to(dev) for x in torch.linalg.eigh(AtA[qf].cpu()))
            rhs = Atb[qf] - (AtA[qf] @ m[:, :, None])[:, :, 0]
            y = (V.transpose(1, 2) @ rhs[:, :, None])[:, :, 0]
            y = torch.where((lam[:, 2:] > 0) & (lam >= 0.01 * lam[:, 2:]), y / lam, 0.0)
            v[rf, g] = m + (V @ y[:, :, None])[:, :, 0]
        re = rows[~full]
        if re.numel():
            mine = (lab[re] == g).to(torch.float64)
            corner = torch.stack([torch.stack([_node(x[re] + ((c >> b) & 1), res) for b, x in enumerate((i, j, k))], 1)
                                  for c in range(8)], 1).to(torch.float64)
            v[re, g] = (corner * mine[:, :, None]).sum(1) / mine.sum(1, keepdim=True)
    out = torch.zeros(6 * res * res, 12, dtype=torch.float64, device=dev)
    out[:keep.numel()] = v[keep].reshape(-1, 12)
    return {"cell": None, "labels, npts, nvert": None, "v": out}


# ---- what a pass cannot do without -----------------------------------------------

def _samples(shape, res):
    """About how many crossings the three images hold: res^2 times the summed
    projected areas of the surface."""
    area = {"sphere": 6 * math.pi * 0.35 ** 2, "flower": 6 * math.pi * 0.3 ** 2,
            "torus": 8 * math.pi * 0.025 + 2 * 16 * 0.025, "knot": 4 * 0.035 * 3.4 * 2.3, "box": 6 * 0.8 ** 2}[shape]
    return area * res * res


def work(case):
    kind = case["kind"]
    if kind == "sample":
        s, rows = _samples(case["shape"], case["res"]), 3 * case["res"] ** 2
        per = 12 if case["packed"] else 20
        return {"bytes": 18 * case["tris"] + 4 * rows + per * s, "flops": 90 * case["tris"] + 12 * s}
    if kind == "frame":
        res = case["res"]
        s, k = _samples("sphere", res), _samples("knot", res)
        return {"bytes": 18 * case["tris"] + 12 * res * res * 4 + 20 * s + 20 * k + 20 * (s + k / 2),
                "flops": 90 * case["tris"] + 20 * (s + k)}
    if kind == "boolean":
        images = 1 if case["api"] == "call" else 3
        s = (_samples(case["a"], case["res"]) + _samples(case["b"], case["res"])) * images / 3
        return {"bytes": 12 * images * case["res"] ** 2 + 20 * s + 14 * s, "flops": 4 * s}
    if kind == "batch":
        by = fl = 0.0
        for m in range(case["count"]):
            tris = case["tris_lo"] * (case["tris_hi"] / case["tris_lo"]) ** ((m * 0.6180339887) % 1.0)
            res = max(64, case["res_hi"] >> ((m * 5 + 3) % 4))
            s = 1.7 * res * res
            by, fl = by + 18 * tris + 12 * res * res + 20 * s, fl + 90 * tris + 12 * s
        return {"bytes": by, "flops": fl}
    if kind == "chain":
        rows = 3 * case["res"] ** 2
        s = case["parts"] * (8 * math.pi * 0.004 + 2 * 16 * 0.004) * case["res"] ** 2
        return {"bytes": 4 * rows * (case["parts"] + 1) + 4 * s + 20 * s / 4, "flops": 2 * s}
    if kind == "gradient":
        s = _samples("sphere", case["res"])
        return {"bytes": 24 * case["tris"] + 12 * case["res"] ** 2 + 20 * s + 8 * s, "flops": 90 * case["tris"] + 60 * s}
    if kind == "nodes":
        s = _samples("sphere", case["res"])
        return {"bytes": 12 * case["res"] ** 2 + 4 * s + case["res"] ** 3 / 8, "flops": 4 * s}
    if kind == "contour":
        s = _samples("sphere", case["res"])  # about as many cells as crossings
        return {"bytes": 12 * case["res"] ** 2 + 20 * s + 72 * s, "flops": 400 * s}
    s = _samples("flower", case["res"])
    return {"bytes": 24 * case["res"] ** 2 + 20 * s + 20 * s, "flops": s * 3 * math.pi * case["radius"] ** 2 * 10}
