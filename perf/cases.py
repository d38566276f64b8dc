"""The work this library is timed on: what a program that simplifies meshes asks of it.

A case is one call, or the few calls of one iteration, through the package's public entry
points (`engine.Context`, `autograd`, `stages`): optimization steps, image losses with their
gradients, reference renders and the per-stage chain, at the sizes, options and meshes of
this repository's workloads and tests (one view of 256x256 up to sixteen of 1024x1024, 300
to a million triangles, maps of 64x64 to 2048x2048, odd image sizes among them).

`exact` restates the renderer in plain torch: visibility by its float32 / int64 contract,
everything else in 64 bits, gradients by reverse-mode differentiation.
"""

import json
import math
import zlib
from types import SimpleNamespace

import numpy as np
import torch

from paper_2104_03989_gb300 import autograd, binding, engine, stages

MAPS = ("kd", "orm", "nrm")
FOVY, NEAR, FAR = 45.0, 0.1, 100.0
F64 = torch.float64
EMPTY = torch.iinfo(torch.int64).max


# ----------------------------------------------------------------------------- cases

def _case(name, call, mesh, n, views, h, w, kd, orm, nrm, loss="logl1", **more):
    """mesh "sphere": 8 n^2 triangles, "quads": 2 n triangles; kd, orm, nrm: sides of the square maps."""
    return {"name": name, "call": call, "mesh": mesh, "n": n, "views": views, "h": h, "w": w, "kd": kd, "orm": orm,
            "nrm": nrm, "loss": loss, **more}


def listed():
    return [
        # the smallest iteration: a 300-triangle sphere under one view; launches and latency are the time
        _case("step_small", "step", "sphere", 6, 1, 256, 256, 256, 1, 256, loss="l1"),
        # the method's ordinary iteration (loss, gradients, Adam) as its loop replays it: one recorded graph
        _case("step_plain", "graph", "sphere", 25, 8, 512, 512, 1024, 1024, 1024),
        # large maps under few small views: the optimizer's pass over the texels is most of the iteration
        _case("step_textures", "step", "sphere", 25, 4, 256, 256, 2048, 2048, 2048),
        # several users' jobs of uneven sizes in one call per stage, as the request loop issues them
        _case("step_jobs", "jobs", "sphere", 16, 6, 256, 256, 512, 512, 512, jobs=8),
        # an odd image size and maps of three different sizes, squared error, gradients for the caller's own optimizer
        _case("grad_ragged", "grad", "sphere", 34, 5, 333, 501, 512, 128, 256, loss="l2"),
        # a base mesh split three times and displaced, sixteen views of 1024x1024: the largest iteration
        _case("grad_tess", "grad", "sphere", 11, 16, 1024, 1024, 1, 1, 2048, tess=3, disp=1024, direct_px=512),
        # multisample antialiasing
        _case("grad_msaa", "grad", "sphere", 25, 8, 512, 512, 1024, 1024, 1024, samples=2),
        # translucent billboards with eight peeled layers: the aggregate-geometry application
        _case("grad_peel", "grad", "quads", 5500, 8, 512, 512, 2048, 1024, 1024, loss="l2", layers=8),
        # an animated mesh: dense weights to 32 bones, a pose per call
        _case("grad_skin", "grad", "sphere", 25, 8, 512, 512, 1024, 1024, 1024, bones=32),
        # the high-poly model's images that every iteration is compared with
        _case("reference_mesh", "reference", "sphere", 158, 8, 512, 512, 2048, 2048, 2048),
        # the same for foliage: six hundred thousand leaf quads, a hundred fragments on a pixel
        _case("reference_leaves", "reference", "quads", 600000, 8, 512, 512, 2048, 2048, 2048, direct_px=256,
              depth_filter=True),
        # the renderer's differentiable stages chained by torch's autograd
        _case("stages_plain", "stages", "sphere", 25, 4, 512, 512, 1024, 1024, 1024),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["step", "step", "graph", "jobs", "grad", "grad", "reference", "stages", "tess", "msaa", "peel",
                       "skin"])
    h = _log(rng, 150, 1024)
    w = h if rng.random() < 0.5 else min(1024, max(150, int(h * rng.uniform(0.6, 1.6))))
    views = min(_log(rng, 1, 16), max(1, 3_000_000 // (h * w)))
    same = rng.random() < 0.6  # the three maps of one size
    kd, orm, nrm = (2 ** rng.randint(6, 11) for _ in range(3))
    if same:
        orm = nrm = kd
    c = _case("", call, "sphere", _log(rng, 6, 50), views, h, w, kd, orm, nrm, loss=rng.choice(["logl1", "l1", "l2"]))
    del c["name"]
    if call == "jobs":
        c.update(jobs=rng.randint(2, 8), views=min(views, 6), h=min(h, 400), w=min(w, 400), kd=min(kd, 512),
                 orm=min(orm, 512), nrm=min(nrm, 512), n=min(c["n"], 30))
    elif call == "reference":
        c["n"] = _log(rng, 25, 160)
    elif call == "tess":
        c.update(call="grad", n=_log(rng, 4, 11), tess=rng.randint(1, 3), disp=2 ** rng.randint(6, 10),
                 direct_px=rng.choice([0, 64, 512]))
    elif call == "msaa":
        c.update(call="grad", samples=rng.randint(2, 3), views=max(1, views // 4))
    elif call == "peel":
        c.update(call="grad", mesh="quads", n=_log(rng, 300, 6000), layers=rng.randint(2, 8), views=max(1, views // 2))
    elif call == "skin":
        c.update(call="grad", bones=_log(rng, 2, 64))
    return c


# ----------------------------------------------------------------------------- inputs

def _sphere(n, bumps):
    """Octahedral sphere of 8 n^2 triangles, tilted off the uv poles; per-corner equirectangular uv (u wraps)."""
    i, j = (a.reshape(-1) for a in np.meshgrid(np.arange(n + 1), np.arange(n + 1), indexing="ij"))
    i, j = i[i + j <= n], j[i + j <= n]
    at = np.full((n + 2, n + 2), -1)
    at[i, j] = np.arange(len(i))
    up = np.stack([at[i, j], at[i + 1, j], at[i, j + 1]], 1)[i + j < n]
    down = np.stack([at[i + 1, j], at[i + 1, j + 1], at[i, j + 1]], 1)[i + j < n - 1]
    face = np.concatenate([up, down])
    pts, tris = [], []
    for k, s in enumerate(np.array([(x, y, z) for x in (1, -1) for y in (1, -1) for z in (1, -1)])):
        pts.append(np.stack([i, j, n - i - j], 1) * s)
        tris.append((face if s.prod() > 0 else face[:, ::-1]) + k * len(i))
    p, back = np.unique(np.concatenate(pts), axis=0, return_inverse=True)
    tri = back.reshape(-1)[np.concatenate(tris)]
    p = p / np.linalg.norm(p, axis=1, keepdims=True)
    ca, sa, cb, sb = math.cos(0.31), math.sin(0.31), math.cos(0.17), math.sin(0.17)
    p = p @ (np.array([[cb, -sb, 0], [sb, cb, 0], [0, 0, 1]]) @ np.array([[1, 0, 0], [0, ca, -sa], [0, sa, ca]])).T
    u, v = np.arctan2(p[:, 2], p[:, 0]) / (2 * np.pi) + 0.5, np.arccos(np.clip(p[:, 1], -1, 1)) / np.pi
    cu, cv = u[tri], v[tri]
    seam = cu.max(1, keepdims=True) - cu.min(1, keepdims=True) > 0.5
    cu = np.where(seam & (cu < 0.5), cu + 1, cu)
    uv = np.stack([cu, cv], 2).reshape(-1, 2)
    d, f, phi = bumps
    p = p * (1 + 0.05 / len(f) * np.sin(f * (p @ d.T) + phi).sum(1, keepdims=True))
    return p, tri, uv, np.arange(3 * len(tri)).reshape(-1, 3)


def _quads(n, rng, lo, hi):
    """n planar quads in an ellipsoid, random orientation, half-sides in [lo, hi], a texture cell each."""
    def unit(k):
        d = rng.normal(size=(k, 3))
        return d / np.linalg.norm(d, axis=1, keepdims=True)

    c = unit(n) * rng.uniform(size=(n, 1)) ** (1 / 3) * np.array([0.9, 0.7, 0.9])
    a, b = unit(n), unit(n)
    b = b - (a * b).sum(1, keepdims=True) * a
    b /= np.linalg.norm(b, axis=1, keepdims=True)
    r = rng.uniform(lo, hi, size=(n, 1))
    a, b = a * r, b * r
    p = np.stack([c - a - b, c + a - b, c + a + b, c - a + b], 1).reshape(-1, 3)
    side = math.ceil(math.sqrt(n))
    k = np.arange(n)
    x0, y0 = (k % side + 0.1) / side, (k // side + 0.1) / side
    x1, y1 = x0 + 0.8 / side, y0 + 0.8 / side
    uv = np.stack([np.stack(q, 1) for q in ((x0, y0), (x1, y0), (x1, y1), (x0, y1))], 1).reshape(-1, 2)
    tri = (4 * k[:, None] + np.array([0, 1, 2, 0, 2, 3])).reshape(-1, 3)
    return p, tri, uv, tri


def _views(rng, n, w, h):
    """Random cameras around the origin, a point and a directional light each: (n, 28) float32 adms_view records."""
    def unit():
        d = rng.normal(size=3)
        return d / np.linalg.norm(d)

    out = np.zeros((n, 28), np.float32)
    t = 1 / math.tan(math.radians(FOVY) / 2)
    proj = np.array([[t * h / w, 0, 0, 0], [0, t, 0, 0],
                     [0, 0, (FAR + NEAR) / (NEAR - FAR), 2 * FAR * NEAR / (NEAR - FAR)], [0, 0, -1, 0]])
    for k in range(n):
        e = unit()
        eye, f = e * rng.uniform(2.5, 4.0), -e
        s = np.cross(f, (0, 1, 0) if abs(f[1]) < 0.999 else (0, 0, 1))
        s /= np.linalg.norm(s)
        look = np.eye(4)
        look[:3, :3] = np.stack([s, np.cross(s, f), -f])
        look[:3, 3] = -look[:3, :3] @ eye
        out[k, :16] = (proj @ look).reshape(-1)
        out[k, 16:19] = eye
        out[k, 20:23], out[k, 23] = unit() * 4.0, 20.0
        out[k, 24:27], out[k, 27] = unit(), 1.0
    return out


def _photos(views, h, w, bumps, dev):
    """What the views see of a lit, patterned unit sphere: reference images (B, h, w, 3) on a black background."""
    v = torch.from_numpy(views).to(dev)
    m = v[:, :16].reshape(-1, 4, 4)
    y, x = torch.meshgrid(torch.arange(h, device=dev) + 0.5, torch.arange(w, device=dev) + 0.5, indexing="ij")
    out = []
    for k in range(len(v)):
        # rows of the MVP: clip.x = t x_cam, clip.y = t y_cam, clip.w = depth along the view
        cx, cy, cw = m[k, 0, :3], m[k, 1, :3], m[k, 3, :3]
        d = (((2 * x / w - 1) / (cx * cx).sum())[..., None] * cx + ((1 - 2 * y / h) / (cy * cy).sum())[..., None] * cy
             + cw)
        d = d / d.norm(dim=-1, keepdim=True)
        eye = v[k, 16:19]
        b = (d * eye).sum(-1)
        disc = b * b - (eye * eye).sum() + 1
        p = eye + (-b - disc.clamp(min=0).sqrt())[..., None] * d
        pat = 0.45 + 0.2 * torch.stack([torch.sin(float(6 * bumps[1][c]) * (p @ torch.from_numpy(
            bumps[0][c]).to(dev, torch.float32)) + float(bumps[2][c])) for c in range(3)], -1)
        lp = v[k, 20:23] - p
        r2 = (lp * lp).sum(-1)
        e = 20 / r2 * ((p * lp).sum(-1) / r2.sqrt()).clamp(min=0) + (p @ v[k, 24:27]).clamp(min=0)
        out.append(torch.where((disc > 0)[..., None], pat * e[..., None] / math.pi, torch.zeros_like(p)))
    return torch.stack(out).contiguous()


def _maps(gen, dev, kd, orm, nrm, smooth, alpha):
    """Base colour (+ opacity), (gamma, r, m) and normal maps: uniform noise (a start of the optimization), or
    smooth ones (an artist's)."""
    def noise(res):
        if not smooth or res < 32:
            return torch.rand(res, res, 4, generator=gen, device=dev)
        t = torch.rand(1, 4, res // 16, res // 16, generator=gen, device=dev)
        return torch.nn.functional.interpolate(t, size=(res, res), mode="bilinear")[0].permute(1, 2, 0).contiguous()

    k, o, n = noise(kd), noise(orm), noise(nrm)
    if alpha:
        k[..., 3] = 0.5
    o[..., 1] = 0.08 + 0.92 * o[..., 1]
    n[..., :2] = (2 * n[..., :2] - 1) * (0.3 if smooth else 1.0)
    if smooth:
        n[..., 2] = 1.0
    o[..., 3] = n[..., 3] = 0.0
    return {"kd": k, "orm": o, "nrm": n}


def _problem(case, seed, dev):
    """One job's inputs: mesh and options on the host, maps and reference images on the device."""
    tag = zlib.crc32(json.dumps({k: v for k, v in case.items() if k != "name"}, sort_keys=True).encode())
    rng = np.random.default_rng([seed, tag])
    gen = torch.Generator(device=dev).manual_seed(int(rng.integers(1 << 62)))
    d = rng.normal(size=(8, 3))
    bumps = (d / np.linalg.norm(d, axis=1, keepdims=True), rng.uniform(2, 8, 8), rng.uniform(0, 2 * np.pi, 8))
    ref = case["call"] == "reference"
    if case["mesh"] == "sphere":
        p, tri, uv, tri_uv = _sphere(case["n"], bumps)
    else:
        p, tri, uv, tri_uv = _quads(case["n"], rng, *((0.015, 0.03) if ref else (0.08, 0.16)))
    q = SimpleNamespace(pos=p.astype(np.float32), tri=tri.astype(np.int32), uv=uv.astype(np.float32),
                        tri_uv=tri_uv.astype(np.int32), views=_views(rng, case["views"], case["w"], case["h"]))
    q.maps = _maps(gen, dev, case["kd"], case["orm"], case["nrm"], ref, case.get("layers", 0) > 0)
    q.ref = None if ref else _photos(q.views, case["h"], case["w"], bumps, dev)
    q.optimize = {"pos": True, **{k: case[k] > 1 for k in MAPS}, "disp": case.get("tess", 0) > 0}
    q.disp = q.weights = q.bones = None
    if case.get("tess", 0):
        q.disp = (torch.rand(case["disp"], case["disp"], generator=gen, device=dev) - 0.5) * 0.02
    if case.get("bones", 0):
        nb = case["bones"]
        # a vertex follows the bones near it; the pose bends each a little
        c = rng.normal(size=(nb, 3))
        g = np.exp(-((p[:, None] - 0.8 * c / np.linalg.norm(c, axis=1, keepdims=True)) ** 2).sum(2) / 0.2) + 1e-4
        q.weights = (g / g.sum(1, keepdims=True)).astype(np.float32)
        q.bones = np.tile(np.eye(4, dtype=np.float32), (nb, 1, 1))
        q.bones[:, :3] += rng.uniform(-0.06, 0.06, size=(nb, 3, 4)).astype(np.float32)
    return q


def _job_cases(case):
    """The uneven jobs of one batched call."""
    out = []
    for k in range(case["jobs"]):
        g = {**case, "call": "step", "n": max(4, case["n"] * (k % 4 + 2) // 4), "views": max(1, case["views"] - k % 3),
             "h": case["h"] * (1 + k % 2), "w": case["w"] * (1 + k % 2), "job": k}
        g.update({m: max(64, case[m] >> (k % 3)) for m in MAPS})
        out.append(g)
    return out


# ----------------------------------------------------------------------------- one pass

def _job(ctx, case, q):
    scene = SimpleNamespace(mesh=SimpleNamespace(pos=q.pos, uv=q.uv, tri_pos=q.tri, tri_uv=q.tri_uv),
                            **{k: q.maps[k].cpu().numpy() for k in MAPS},
                            disp=None if q.disp is None else q.disp.cpu().numpy(), tess_levels=case.get("tess", 0),
                            mips=True, optimize=q.optimize)
    job = ctx.create_job(scene, loss=case["loss"], lr0=0.01, frozen=case["call"] == "reference",
                         samples=case.get("samples", 1), layers=case.get("layers", 0),
                         raster_direct_px=case.get("direct_px", 0),
                         raster_depth_filter=case.get("depth_filter", False))
    if q.weights is not None:
        ctx.skinning(job, q.weights, lr_scale=1.0 / q.weights.shape[1])
    return job


def _latents(ctx, job, q):
    p = ctx.params(job)
    out = {"pos": p["pos"], **{k: p[k + "_chain"] for k in MAPS if q.optimize[k]}}
    for t in out.values():
        t.owner = ctx  # the memory is the context's: it lives as long as what is returned of it
    return out


def prepare(case, seed):
    if case["call"] == "stages":
        q = _problem(case, seed, "cuda")
        leaf = {"pos": torch.from_numpy(q.pos).cuda().requires_grad_(True),
                **{k: q.maps[k].requires_grad_(True) for k in MAPS}}
        pipe = stages.Pipeline(q.tri, q.uv, q.tri_uv, len(q.pos), q.views, case["h"], case["w"])
        return {"call": "stages", "pipe": pipe, "leaf": leaf, "ref": q.ref, "loss": case["loss"]}
    graph = case["call"] == "graph"
    ctx = engine.Context(stream=torch.cuda.Stream() if graph else None)
    qs = [_problem(c, seed, "cuda") for c in (_job_cases(case) if case["call"] == "jobs" else [case])]
    torch.cuda.synchronize()
    s = {"call": case["call"], "ctx": ctx, "jobs": [_job(ctx, case, q) for q in qs], "views": [q.views for q in qs],
         "refs": [q.ref for q in qs], "size": (case["h"], case["w"])}
    if case["call"] == "grad":
        names = ["pos"] + [k for k in MAPS if qs[0].optimize[k]]
        names += (["disp"] if case.get("tess", 0) else []) + (["w"] if case.get("bones", 0) else [])
        s["leaf"] = autograd.latents(ctx, s["jobs"][0], names)
        s["bones"] = None if qs[0].bones is None else torch.from_numpy(qs[0].bones).cuda()
    elif case["call"] != "reference":
        s["latents"] = [_latents(ctx, j, q) for j, q in zip(s["jobs"], qs)]
    if graph:
        # the loop's step recorded once: fixed buffers for the views, the reference images and the loss
        job, views = s["jobs"][0], torch.from_numpy(qs[0].views).cuda()
        s["loss"] = torch.zeros(1, device="cuda")
        ctx.reserve(job, case["views"], case["h"], case["w"])
        torch.cuda.synchronize()
        binding.adms_graph_begin(ctx.ctx)
        binding.adms_forward_loss(ctx.ctx, [job], views, [case["views"]], [s["size"]], s["refs"], s["loss"])
        ctx.backward([job])
        ctx.step([job])
        s["graph"], s["recorded"] = binding.adms_graph_end(ctx.ctx), views
    return s


def run(s):
    call = s["call"]
    if call == "stages":
        lf = s["leaf"]
        loss = stages.render_loss(s["pipe"], lf["pos"], lf["kd"], lf["orm"], lf["nrm"], s["ref"], s["loss"])
        return {"loss": loss.detach(), "grad": dict(zip(lf, torch.autograd.grad(loss, list(lf.values()))))}
    ctx = s["ctx"]
    if call == "graph":
        binding.adms_graph_launch(ctx.ctx, s["graph"])
        return {"loss": s["loss"], "job0": s["latents"][0]}
    if call in ("step", "jobs"):
        loss = ctx.forward_loss(s["jobs"], s["views"], s["refs"])
        ctx.backward(s["jobs"])
        ctx.step(s["jobs"])
        return {"loss": loss, **{"job%d" % k: v for k, v in enumerate(s["latents"])}}
    if call == "reference":
        return {"image": ctx.render_reference(s["jobs"][0], s["views"][0], *s["size"])}
    autograd.invalidate(ctx, s["jobs"][0])  # the caller's optimizer has written the latents since the last pass
    if s["bones"] is not None:
        ctx.set_bones(s["jobs"][0], s["bones"])
    loss = autograd.render_loss(ctx, s["jobs"][0], s["views"][0], s["refs"][0], s["leaf"])
    return {"loss": loss.detach(), "grad": dict(zip(s["leaf"], torch.autograd.grad(loss, list(s["leaf"].values()))))}


# ----------------------------------------------------------------------------- work

def work(case):
    if case["call"] == "jobs":
        ws = [work(c) for c in _job_cases(case)]
        return {k: sum(w[k] for w in ws) for k in ws[0]}
    px = case["views"] * case["h"] * case["w"]
    if case["mesh"] == "sphere":  # the disc of a unit sphere seen from 2.5 to 4, 45 degrees high
        cover = 0.46 * min(1.0, case["h"] / case["w"])
        tris = 8 * case["n"] ** 2
        verts = tris // 2 + 2
        frags = cover * px * case.get("samples", 1) ** 2
    else:
        cover, tris, verts = 0.35 * min(1.0, case["h"] / case["w"]), 2 * case["n"], 4 * case["n"]
        frags = cover * px * case.get("layers", 1)
    base_verts = verts
    if case.get("tess", 0):
        tris *= 4 ** case["tess"]
    texels = {k: case[k] ** 2 for k in MAPS}
    read = {k: min(texels[k] * 4 / 3, 4 / 3 * frags) for k in MAPS}
    mesh = 12 * verts + 24 * tris + 8 * 3 * tris
    if case["call"] == "reference":
        return {"bytes": mesh + 16 * sum(read.values()) + 12 * px, "flops": 700 * frags}
    opt = [k for k in MAPS if case[k] > 1]
    b = mesh + 12 * px + 16 * sum(read.values())
    if case["call"] in ("step", "graph"):
        # latent and two moments read and written, the coarser levels written
        b += sum(16 * texels[k] * (6 + 1 / 3) for k in opt) + 12 * 6 * base_verts
    else:
        b += sum(16 * texels[k] for k in opt) + 12 * base_verts
        b += 2 * 4 * case.get("disp", 0) ** 2 + 3 * 4 * base_verts * case.get("bones", 0)
    return {"bytes": b, "flops": 2200 * frags + 40 * px}


# ----------------------------------------------------------------------------- the same in 64 bits

def _unit(x):
    return x / (x * x).sum(-1, keepdim=True).clamp(min=1e-20).sqrt()


def _dot(a, b):
    return (a * b).sum(-1, keepdim=True)


def _cross2(a, b):
    return a[..., 0] * b[..., 1] - a[..., 1] * b[..., 0]


def _chain(t):
    """(texels, 4) of all levels of the box-filter chain, and the levels' (offset, h, w)."""
    lv = [t]
    while max(lv[-1].shape[:2]) > 1:
        h, w, c = lv[-1].shape
        sh, sw = min(h, 2), min(w, 2)
        lv.append(lv[-1].reshape(h // sh, sh, w // sw, sw, c).mean(dim=(1, 3)))
    at, offs = 0, []
    for x in lv:
        offs.append((at, x.shape[0], x.shape[1]))
        at += x.shape[0] * x.shape[1]
    return torch.cat([x.reshape(-1, x.shape[2]) for x in lv]), offs


def _bilinear(flat, off, h, w, uv):
    """Bilinear lookup in levels of `flat` (u wraps, v clamps); off, h, w: per lookup."""
    x, y = uv[:, 0] * w - 0.5, uv[:, 1] * h - 0.5
    x0, y0 = x.detach().floor(), y.detach().floor()
    fx, fy = (x - x0)[:, None], (y - y0)[:, None]
    xi, yi = x0.long(), y0.long()
    xa, xb = torch.remainder(xi, w), torch.remainder(xi + 1, w)
    ya, yb = torch.minimum(yi.clamp(min=0), h - 1), torch.minimum((yi + 1).clamp(min=0), h - 1)

    def at(yy, xx):
        return flat.index_select(0, off + yy * w + xx)

    return (1 - fy) * ((1 - fx) * at(ya, xa) + fx * at(ya, xb)) + fy * ((1 - fx) * at(yb, xa) + fx * at(yb, xb))


def _trilinear(flat, offs, uv, dx, dy):
    o = torch.tensor(offs, device=uv.device)
    wh = torch.tensor([offs[0][2], offs[0][1]], dtype=F64, device=uv.device)
    rho = torch.maximum((dx * wh).norm(dim=1), (dy * wh).norm(dim=1))
    lod = torch.nan_to_num(torch.log2(rho), nan=0.0, neginf=0.0).clamp(0, len(offs) - 1).detach()
    l0 = lod.floor().long()
    fr = (lod - l0)[:, None]
    out = 0.0
    for k, wl in ((l0, 1 - fr), ((l0 + 1).clamp(max=len(offs) - 1), fr)):
        out = out + wl * _bilinear(flat, o[k, 0], o[k, 1], o[k, 2], uv)
    return out


def _around(tri, n):
    """Faces of each vertex in ascending order, padded with the face count: (n, valence)."""
    flat = np.asarray(tri).reshape(-1)
    order = np.argsort(flat, kind="stable")
    count = np.bincount(flat, minlength=n)
    out = np.full((n, max(1, count.max())), len(tri))
    slot = np.arange(len(flat)) - np.repeat(np.cumsum(count) - count, count)
    out[flat[order], slot] = order // 3
    return out


def _tessellate(tri, tri_uv, uv, levels):
    """The lattice of 2^levels segments per edge: render triangles, uv corners, and each vertex's base triangle and
    integer weights (a shared vertex belongs to the lowest-numbered face)."""
    n, faces = 1 << levels, len(tri)
    i, j = (a.reshape(-1) for a in np.meshgrid(np.arange(n + 1), np.arange(n + 1), indexing="ij"))
    i, j = i[i + j <= n], j[i + j <= n]
    at = np.full((n + 2, n + 2), -1)
    at[i, j] = np.arange(len(i))
    wt = np.stack([n - i - j, i, j], 1)
    cells = []
    for a in range(n):
        for b in range(n - a):
            cells.append((at[a, b], at[a + 1, b], at[a, b + 1]))
            if a + b + 1 < n:
                cells.append((at[a + 1, b], at[a + 1, b + 1], at[a, b + 1]))
    cells = np.array(cells)
    far = tri.max() + 1
    ids = np.where(wt[None] > 0, tri[:, None, :], far).astype(np.int64)
    order = np.argsort(ids, 2, kind="stable")
    ids, ws = np.take_along_axis(ids, order, 2), np.take_along_axis(np.broadcast_to(wt, ids.shape), order, 2)
    key = np.concatenate([ids, ws], 2).reshape(-1, 6)
    key = ((((key[:, 0] * (far + 1) + key[:, 1]) * (far + 1) + key[:, 2]) * (n + 1)) + key[:, 3]) * (n + 1) + key[:, 4]
    _, first, back = np.unique(key, return_index=True, return_inverse=True)
    rank = np.argsort(np.argsort(first))  # vertices numbered by first occurrence
    first = np.sort(first)
    g = rank[back.reshape(-1)].reshape(faces, -1)
    corner = (wt[None, :, :, None] / n * uv[tri_uv][:, None]).sum(2)
    return SimpleNamespace(tri=g[:, cells].reshape(-1, 3), uv=corner.reshape(-1, 2).astype(np.float32),
                           tri_uv=(np.arange(faces)[:, None, None] * len(i) + cells[None]).reshape(-1, 3),
                           owner=tri[first // len(i)].astype(np.int64), wts=wt[first % len(i)],
                           at=corner.reshape(-1, 2)[first].astype(np.float32), n=n)


def _displaced(pos, disp, tri, tess, f32):
    """Eq. 3 positions of the render mesh; in float32 by the visibility's contract (each operation rounded once, in
    this order), else in 64 bits."""
    dev = pos.device
    ty = torch.float32 if f32 else F64
    p, dm = pos.to(ty), disp.to(ty)
    t = torch.from_numpy(np.asarray(tri, np.int64)).to(dev)
    e1, e2 = p[t[:, 1]] - p[t[:, 0]], p[t[:, 2]] - p[t[:, 0]]
    fn = torch.stack([e1[:, 1] * e2[:, 2] - e1[:, 2] * e2[:, 1], e1[:, 2] * e2[:, 0] - e1[:, 0] * e2[:, 2],
                      e1[:, 0] * e2[:, 1] - e1[:, 1] * e2[:, 0]], 1)
    fn = torch.cat([fn, torch.zeros_like(fn[:1])])
    inc = torch.from_numpy(_around(tri, len(pos))).to(dev)
    s = torch.zeros_like(p)
    for k in range(inc.shape[1]):
        s = s + fn[inc[:, k]]

    def norm(x):
        return ((x[:, 0] * x[:, 0] + x[:, 1] * x[:, 1]) + x[:, 2] * x[:, 2]).clamp(min=1e-20).sqrt()[:, None]

    nrm = s / norm(s)
    o, w = torch.from_numpy(tess.owner).to(dev), torch.from_numpy(tess.wts).to(dev, ty) / torch.tensor(
        float(tess.n), dtype=ty, device=dev)

    def mix(a):
        return (w[:, 0:1] * a[o[:, 0]] + w[:, 1:2] * a[o[:, 1]]) + w[:, 2:3] * a[o[:, 2]]

    v, ns = mix(p), mix(nrm)
    uv = torch.from_numpy(tess.at).to(dev, ty)
    h, wd = disp.shape
    x, y = uv[:, 0] * wd - 0.5, uv[:, 1] * h - 0.5
    x0, y0 = x.floor(), y.floor()
    fx, fy = x - x0, y - y0
    xa, ya = torch.remainder(x0.long(), wd), y0.long()
    xb, yb, ya = torch.remainder(xa + 1, wd), (ya + 1).clamp(0, h - 1), ya.clamp(0, h - 1)
    gx, gy = 1 - fx, 1 - fy
    d = ((gx * gy) * dm[ya, xa] + (fx * gy) * dm[ya, xb]) + ((gx * fy) * dm[yb, xa] + (fx * fy) * dm[yb, xb])
    return v + d[:, None] * (ns / norm(ns))


def _skinned(pos, weights, bones, f32):
    """Eq. 2; in float32 by the visibility's contract (bones ascending), else in 64 bits."""
    ty = torch.float32 if f32 else F64
    p, w, m = pos.to(ty), weights.to(ty), bones.to(ty)
    out = torch.zeros_like(p)
    for b in range(m.shape[0]):
        t = [((m[b, r, 0] * p[:, 0] + m[b, r, 1] * p[:, 1]) + m[b, r, 2] * p[:, 2]) + m[b, r, 3] for r in range(3)]
        out = out + w[:, b:b + 1] * torch.stack(t, 1)
    return out


def _frame(pos, tri, uv, tri_uv):
    """Unit smooth normals and tangents of the vertices."""
    p0, p1, p2 = (pos[tri[:, k]] for k in range(3))
    t0, t1, t2 = (uv[tri_uv[:, k]] for k in range(3))
    e1, e2, d1, d2 = p1 - p0, p2 - p0, t1 - t0, t2 - t0
    fn = torch.linalg.cross(e1, e2, dim=1)
    ft = _unit(e1 * d2[:, 1:2] - e2 * d1[:, 1:2]) * torch.sign(_cross2(d1, d2))[:, None]
    n, t = torch.zeros_like(pos), torch.zeros_like(pos)
    for k in range(3):
        n, t = n.index_add(0, tri[:, k], fn), t.index_add(0, tri[:, k], ft)
    return _unit(n), _unit(t)


def _neighbours(tri):
    """The face across each edge (a, b), (b, c), (c, a), or -1."""
    t = np.asarray(tri, np.int64)
    a, b = t[:, [0, 1, 2]].reshape(-1), t[:, [1, 2, 0]].reshape(-1)
    key = np.minimum(a, b) * (t.max() + 1) + np.maximum(a, b)
    order = np.argsort(key, kind="stable")
    ks = key[order]
    start = np.concatenate([[True], ks[1:] != ks[:-1]])
    group = np.cumsum(start) - 1
    size = np.bincount(group)[group]
    first = np.flatnonzero(start)[group]
    other = np.where(np.arange(len(ks)) == first, np.minimum(first + 1, len(ks) - 1), first)
    out = np.full(len(key), -1, np.int64)
    out[order] = np.where(size == 2, order[other] // 3, -1)
    return out.reshape(-1, 3)


def _visible(p32, tri, m, h, w, layers):
    """Depth | id keys of the nearest `layers` fragments of each sample of one view, and the triangles' area signs."""
    dev = p32.device
    x, y, z = p32.unbind(1)
    c = [((m[4 * r] * x + m[4 * r + 1] * y) + m[4 * r + 2] * z) + m[4 * r + 3] for r in range(4)]
    hw, hh = (torch.tensor(0.5 * v, dtype=torch.float32, device=dev) for v in (w, h))
    sx, sy = c[0] / c[3] * hw + hw, hh - c[1] / c[3] * hh
    fx, fy = sx * 256, sy * 256
    ok = (c[3] > 1e-6) & (fx.abs() <= 134217728.0) & (fy.abs() <= 134217728.0)
    X, Y = (torch.where(ok, v, torch.zeros_like(v)).round().long() for v in (fx, fy))
    Z = c[2] / c[3] * 0.5 + 0.5
    T = [[X[tri[:, k]], Y[tri[:, k]]] for k in range(3)]
    area = (T[1][0] - T[0][0]) * (T[2][1] - T[0][1]) - (T[1][1] - T[0][1]) * (T[2][0] - T[0][0])
    area = torch.where(ok[tri].all(1), area, torch.zeros_like(area))
    sign = torch.sign(area)
    lo = [torch.minimum(torch.minimum(T[0][k], T[1][k]), T[2][k]) for k in (0, 1)]
    hi = [torch.maximum(torch.maximum(T[0][k], T[1][k]), T[2][k]) for k in (0, 1)]
    i0, j0 = (torch.div(v + 127, 256, rounding_mode="floor").clamp(min=0) for v in lo)
    i1, j1 = (torch.minimum(torch.div(v - 128, 256, rounding_mode="floor"), torch.tensor(e - 1, device=dev))
              for v, e in zip(hi, (w, h)))
    nx, ny = (i1 - i0 + 1).clamp(min=0), (j1 - j0 + 1).clamp(min=0)
    count = torch.where(area != 0, nx * ny, torch.zeros_like(nx))
    live = torch.nonzero(count)[:, 0]
    keys = torch.full((layers, h * w), EMPTY, dtype=torch.int64, device=dev)
    ends = count[live].cumsum(0)
    total = int(ends[-1]) if len(live) else 0
    cuts = torch.searchsorted(ends, torch.arange(0, total, 1 << 24, device=dev), right=True).tolist() + [len(live)]
    found = []
    for a, b in zip(cuts[:-1], cuts[1:]):
        f = live[a:b]
        cnt = count[f]
        if not len(f):
            continue
        k = torch.arange(int(cnt.sum()), device=dev) - torch.repeat_interleave(cnt.cumsum(0) - cnt, cnt)
        f = torch.repeat_interleave(f, cnt)
        px, py = i0[f] + k % nx[f], j0[f] + torch.div(k, nx[f], rounding_mode="floor")
        Sx, Sy = 256 * px + 128, 256 * py + 128
        s, hit, E = sign[f], torch.ones_like(f, dtype=torch.bool), []
        for e in range(3):
            (ax, ay), (bx, by) = ((T[(e + q) % 3][0][f], T[(e + q) % 3][1][f]) for q in (1, 2))
            dx, dy = bx - ax, by - ay
            v = dx * (Sy - ay) - dy * (Sx - ax)
            top = (s * dy < 0) | ((dy == 0) & (s * dx > 0))
            hit &= torch.where(top, s * v >= 0, s * v > 0)
            E.append(v)
        f, px, py, fA = f[hit], px[hit], py[hit], area[f][hit].float()
        z0, z1, z2 = (Z[tri[f, q]] for q in range(3))
        d = (z0 + E[1][hit].float() / fA * (z1 - z0)) + E[2][hit].float() / fA * (z2 - z0)
        good = (d >= 0) & (d <= 1)
        d = torch.where(d == 0, torch.zeros_like(d), d)
        found.append((py[good] * w + px[good], (d[good].contiguous().view(torch.int32).long() << 32) | f[good]))
    for layer in range(layers):
        for at, key in found:
            if layer:
                deeper = key > keys[layer - 1][at]
                at, key = at[deeper], key[deeper]
            keys[layer].scatter_reduce_(0, at, key, "amin")
    return keys, sign


def _shade(g, chains, view, ids, w, s):
    """Colour and opacity of the samples with triangle ids >= 0, and their places."""
    at = torch.nonzero(ids >= 0)[:, 0]
    f = ids[at]
    q = torch.stack([((at % w) // s) * s + 0.5 * s, (torch.div(at, w, rounding_mode="floor") // s) * s + 0.5 * s], 1)
    vi, ui = g.tri[f], g.tri_uv[f]
    sc, cw = [g.scr[vi[:, k]] for k in range(3)], [g.clip[vi[:, k], 3] for k in range(3)]
    area = _cross2(sc[1] - sc[0], sc[2] - sc[0])
    r = [_cross2(sc[(k + 1) % 3] - q, sc[(k + 2) % 3] - q) / area / cw[k] for k in range(3)]
    R = r[0] + r[1] + r[2]
    beta = [x / R for x in r]
    with torch.no_grad():
        duv = []
        for ax, sg in ((1, 1.0), (0, -1.0)):
            dr = [sg * (sc[(k + 1) % 3][:, ax] - sc[(k + 2) % 3][:, ax]) / area / cw[k] for k in range(3)]
            dR = dr[0] + dr[1] + dr[2]
            duv.append(s * sum(((dr[k] * R - r[k] * dR) / (R * R))[:, None] * g.uv[ui[:, k]] for k in range(3)))

    def mix(a, idx):
        return sum(beta[k][:, None] * a[idx[:, k]] for k in range(3))

    p, n, t, uv = mix(g.pos, vi), mix(g.nrm, vi), mix(g.tan, vi), mix(g.uv, ui)
    kd, orm, nm = (_trilinear(*chains[k], uv, *duv) for k in MAPS)
    N = _unit(n)
    T = _unit(t - _dot(t, N) * N)
    ns = _unit(nm[:, 0:1] * T + nm[:, 1:2] * torch.linalg.cross(N, T, dim=1) + nm[:, 2:3] * N)
    V = _unit(view[16:19] - p)
    nv = _dot(ns, V).clamp(min=1e-4)
    a2 = orm[:, 1:2].clamp(min=0.08) ** 4
    gam, m, c3 = orm[:, 0:1], orm[:, 2:3], kd[:, :3]
    ks, diff = (1 - m) * 0.04 + m * c3, c3 * (1 - m) / math.pi

    def g1(c):
        return 2 * c / (c + (a2 + (1 - a2) * c * c).sqrt())

    lp = view[20:23] - p
    col = 0.0
    for L, E in ((_unit(lp), view[23] / _dot(lp, lp)), (view[24:27].expand_as(p), view[27])):
        nl = _dot(ns, L)
        lit = nl > 0
        nl = torch.where(lit, nl, torch.ones_like(nl))
        H = _unit(L + V)
        nh, vh = _dot(ns, H).clamp(min=0), _dot(V, H).clamp(min=0)
        D = a2 / (math.pi * (nh * nh * (a2 - 1) + 1) ** 2)
        F = ks + (1 - ks) * (1 - vh) ** 5
        spec = (1 - gam) * D * F * g1(nl) * g1(nv) / (4 * nl * nv)
        col = col + torch.where(lit, (diff + spec) * E * nl, torch.zeros_like(c3))
    return at, col, kd[:, 3:4]


def _antialias(flat, keys, ids, g, sil, h, w):
    """Silhouette antialiasing of (h w, 3) colours: each pair of neighbours blends by where an edge of the nearer
    triangle's silhouette crosses between their centres."""
    grid = torch.arange(h * w, device=flat.device).reshape(h, w)
    out = flat
    for axis in (0, 1):
        p, q = (grid[:, :-1], grid[:, 1:]) if axis == 0 else (grid[:-1], grid[1:])
        p, q = p.reshape(-1), q.reshape(-1)
        pair = ids[p] != ids[q]
        p, q = p[pair], q[pair]
        if not len(p):
            continue
        near = keys[p] < keys[q]
        o, s = torch.where(near, p, q), torch.where(near, q, p)
        sigma = torch.where(near, 1.0, -1.0).to(F64)
        f = ids[o]
        c = torch.stack([o % w + 0.5, torch.div(o, w, rounding_mode="floor") + 0.5], 1).to(F64)
        ux, xx = (1, 0) if axis == 0 else (0, 1)
        tau = torch.full((len(p),), 0.5, dtype=F64, device=flat.device)
        best = torch.full_like(tau, math.inf)
        for e in range(3):
            a, b = g.scr[g.tri[f, e]], g.scr[g.tri[f, (e + 1) % 3]]
            den = b[:, ux] - a[:, ux]
            sp = (c[:, ux] - a[:, ux]) / torch.where(den != 0, den, torch.ones_like(den))
            t = sigma * (a[:, xx] + sp * (b[:, xx] - a[:, xx]) - c[:, xx])
            take = sil[f, e] & (den != 0) & (sp >= 0) & (sp <= 1) & (t > 0) & (t < 1) & (t < best)
            best, tau = torch.where(take, t.detach(), best), torch.where(take, t, tau)
        move = (tau - 0.5)[:, None]
        co, cs = flat[o], flat[s]
        zero = torch.zeros_like(co)
        out = out.index_add(0, s, torch.where(move > 0, move * (co - cs), zero))
        out = out.index_add(0, o, torch.where(move < 0, -move * (cs - co), zero))
    return out


def _tone(x):
    x = torch.log(x.clamp(min=0) + 1)
    return torch.where(x <= 0.0031308, 12.92 * x, 1.055 * x.clamp(min=0.0031308) ** (1 / 2.4) - 0.055)


def _terms(img, ref, kind):
    if kind == "l2":
        return (img - ref) ** 2
    return (img - ref).abs() if kind == "l1" else (_tone(img) - _tone(ref)).abs()


def _solve(case, seed):
    """The image losses' sum, each latent's gradient (dict), the leaves, the images where no loss is taken."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    q = _problem(case, seed, dev)
    ref = case["call"] == "reference"
    leaf = {"pos": torch.from_numpy(q.pos).to(dev, F64), **{k: q.maps[k].to(F64) for k in MAPS}}
    if q.disp is not None:
        leaf["disp"] = q.disp.to(F64)
    if q.weights is not None:
        leaf["w"] = torch.from_numpy(q.weights).to(dev, F64)
        bones = torch.from_numpy(q.bones).to(dev)
    for k, t in leaf.items():
        t.requires_grad_(not ref and q.optimize.get(k, True))
    tri, uv, tri_uv = q.tri.astype(np.int64), q.uv, q.tri_uv.astype(np.int64)
    pos = leaf["pos"]
    if q.disp is not None:
        t = _tessellate(tri, tri_uv, uv, case["tess"])
        pos = _displaced(pos, leaf["disp"], tri, t, False)
        # the values rendered are the contract's float32 ones, differentiated as the 64-bit expression
        pos = pos + (_displaced(leaf["pos"], leaf["disp"], tri, t, True).to(F64) - pos).detach()
        tri, uv, tri_uv = t.tri, t.uv, t.tri_uv
    if q.weights is not None:
        pos = _skinned(pos, leaf["w"], bones, False)
        pos = pos + (_skinned(leaf["pos"], leaf["w"], bones, True).to(F64) - pos).detach()
    adj = torch.from_numpy(_neighbours(tri)).to(dev)
    g = SimpleNamespace(tri=torch.from_numpy(tri).to(dev), tri_uv=torch.from_numpy(tri_uv).to(dev),
                        uv=torch.from_numpy(uv).to(dev, F64))
    nrm, tan = _frame(pos, g.tri, g.uv, g.tri_uv)
    chains = {k: _chain(leaf[k]) for k in MAPS}
    # the views share leaves below the frame and the chains, so that each view's graph is freed with it
    top = {"pos": pos, "normal": nrm, "tangent": tan, **{k: chains[k][0] for k in MAPS}}
    sub = {k: v.detach().requires_grad_(v.requires_grad) for k, v in top.items()}
    g.pos, g.nrm, g.tan = sub["pos"], sub["normal"], sub["tangent"]
    chains = {k: (sub[k], chains[k][1]) for k in MAPS}
    s, layers = case.get("samples", 1), case.get("layers", 0)
    h, w = case["h"] * s, case["w"] * s
    loss, images = 0.0, []
    for b in range(case["views"]):
        v32 = torch.from_numpy(q.views[b]).to(dev)
        view = v32.to(F64)
        keys, sign = _visible(g.pos.detach().float(), g.tri, v32[:16], h, w, max(layers, 1))
        sil = (adj < 0) | (sign[adj.clamp(min=0)] != sign[:, None])
        g.clip = torch.cat([g.pos, torch.ones_like(g.pos[:, :1])], 1) @ view[:16].reshape(4, 4).T
        hw, hh = 0.5 * w, 0.5 * h
        g.scr = torch.stack([g.clip[:, 0] / g.clip[:, 3] * hw + hw, hh - g.clip[:, 1] / g.clip[:, 3] * hh], 1)
        acc = torch.zeros(h * w, 3, dtype=F64, device=dev)
        for key in keys.flip(0):
            ids = torch.where(key == EMPTY, torch.full_like(key, -1), key & 0xFFFFFFFF)
            at, col, alpha = _shade(g, chains, view, ids, w, s)
            if layers:
                acc = acc.index_copy(0, at, alpha * col + (1 - alpha) * acc[at])
            else:
                acc = torch.zeros_like(acc).index_copy(0, at, col)
            acc = _antialias(acc, key, ids, g, sil, h, w)
        img = acc.reshape(case["h"], s, case["w"], s, 3).mean(dim=(1, 3))
        if ref:
            images.append(img)
            continue
        part = _terms(img, q.ref[b].to(F64), case["loss"]).sum() / (3 * case["views"] * case["h"] * case["w"])
        part.backward()
        loss += float(part.detach())
    if ref:
        return None, None, None, torch.stack(images)
    torch.autograd.backward([top[k] for k in top if top[k].requires_grad],
                            [sub[k].grad if sub[k].grad is not None else torch.zeros_like(sub[k])
                             for k in top if top[k].requires_grad])
    return loss, {k: t.grad for k, t in leaf.items() if t.requires_grad}, leaf, tri


def _stepped(case, seed):
    """One optimizer step from the given latents: the Laplacian term weighted by a quarter of the image loss over
    it, Adam, the ranges, and the chains of the updated maps."""
    loss, grad, leaf, tri = _solve(case, seed)
    pos = leaf["pos"].detach().requires_grad_(True)
    e = np.concatenate([tri[:, [0, 1]], tri[:, [1, 2]], tri[:, [2, 0]]])
    e = torch.from_numpy(np.unique(np.concatenate([e, e[:, ::-1]]), axis=0)).to(pos.device)
    deg = torch.bincount(e[:, 0], minlength=len(pos))[:, None].to(F64)
    delta = pos - torch.zeros_like(pos).index_add(0, e[:, 0], pos[e[:, 1]]) / deg
    lap = (delta * delta).sum(1).mean()
    grad["pos"] = grad["pos"] + 0.25 * loss / float(lap.detach()) * torch.autograd.grad(lap, pos)[0]
    lim = {"kd": ((0, 1),) * 4, "orm": ((0, 1), (0.08, 1), (0, 1), None), "nrm": ((-1, 1), (-1, 1), (0, 1), None)}
    out = {}
    for k, gr in grad.items():
        x = leaf[k].detach() - 0.01 * gr / (gr.abs() + 1e-8)
        if k in MAPS:
            x = torch.stack([x[..., c] if r is None else x[..., c].clamp(*r) for c, r in enumerate(lim[k])], -1)
            x = _chain(x)[0]
        out[k] = x
    return torch.tensor([loss], dtype=F64), out


def exact(case, seed):
    call = case["call"]
    if call == "reference":
        return {"image": _solve(case, seed)[3]}
    if call in ("step", "graph", "jobs"):
        got = [_stepped(c, seed) for c in (_job_cases(case) if call == "jobs" else [case])]
        return {"loss": torch.cat([x[0] for x in got]), **{"job%d" % k: x[1] for k, x in enumerate(got)}}
    loss, grad, _, _ = _solve(case, seed)
    return {"loss": torch.tensor(loss, dtype=F64), "grad": grad}
