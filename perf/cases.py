"""The measured work: what programs that use this framework have it do.

Training steps (one CUDA graph per step, or call by call with the D-SSIM
loss), differentiable renders through torch.autograd, forward renders, a burst
of requests to the render server, and the steps around training: the image
loss, the crossings of a volume, the initial Gaussians of a point cloud and
one densification.  Scenes are isosurfaces of seeded analytic fields with the
sizes of the repository's benchmark workloads; everything is made on the GPU
from the seed.

`exact` restates the mathematics in 64-bit torch (projection, per-tile
compositing by cumulative products, SSIM, Adam, crossings, neighbours,
densification) without this package's code.
"""
from __future__ import annotations

import math
import random

import torch

from paper_2509_05216_gb300 import autograd, gs, inputs

DEV = "cuda"
#: learning rates at the end of a decaying schedule (a hundredth of the start's), so that a state that
#: is stepped many times stays the scene it was
HP = {k: v * 0.01 if k.startswith("lr_") else v for k, v in autograd.Adam.DEFAULTS.items()}
STEP0 = 7000  # steps already taken: the moments are warm
#: orbit radius and half width of the box of each scene
SCENES = {"sphere": (3.0, 1.0), "gyroid": (15.0, 2.0 * math.pi), "blobs": (4.0, 1.0), "noise": (4.0, 1.0)}


def listed():
    return [
        # the smallest training step: 10,000 Gaussians, one small view; latency and launches count
        {"name": "step_sphere_10k", "kind": "step", "scene": "sphere", "n": 10_000, "deg": 0, "views": 1,
         "w": 256, "h": 256},
        # ordinary batched training: half a million Gaussians, 8 views
        {"name": "step_gyroid_500k", "kind": "step", "scene": "gyroid", "n": 500_000, "deg": 3, "views": 8,
         "w": 1024, "h": 1024},
        # the benchmark's training step: 4M Gaussians, 16 views
        {"name": "step_blobs_4m", "kind": "step", "scene": "blobs", "n": 4_000_000, "deg": 3, "views": 16,
         "w": 2048, "h": 2048},
        # the largest training step: 18M Gaussians, 4 large views
        {"name": "step_noise_18m", "kind": "step", "scene": "noise", "n": 18_000_000, "deg": 3, "views": 4,
         "w": 4096, "h": 4096},
        # one view per step, call by call, L1 + D-SSIM, visible-only Adam, from close by (part of the set is
        # out of view), ragged size: how 3D-GS trainers iterate
        {"name": "view_blobs_4m", "kind": "view", "scene": "blobs", "n": 4_000_000, "deg": 3, "views": 1,
         "w": 1919, "h": 1081},
        # a caller's own loss through torch.autograd: few large splats, odd view sizes, degree 2, a background
        {"name": "autograd_37k", "kind": "autograd", "scene": "sphere", "n": 37_001, "deg": 2, "views": 3,
         "w": 517, "h": 333},
        # one large frame of a trained set (interactive viewing)
        {"name": "render_blobs_4m", "kind": "render", "scene": "blobs", "n": 4_000_000, "deg": 3, "views": 1,
         "w": 3840, "h": 2160},
        # a burst of mixed-resolution requests to the render server
        {"name": "serve_blobs_1m", "kind": "serve", "scene": "blobs", "n": 1_000_003, "deg": 3, "views": 12,
         "w": 2048, "h": 2048},
        # the D-SSIM loss and its gradient over a batch
        {"name": "ssim_16x2048", "kind": "ssim", "views": 16, "w": 2048, "h": 2048},
        # contour points and normals of a volume
        {"name": "crossings_512", "kind": "crossings", "nx": 512, "ny": 512, "nz": 512},
        # initial Gaussians of a point cloud, picked from a larger one
        {"name": "init_4m", "kind": "init", "scene": "blobs", "n": 4_000_000, "deg": 3},
        # one densification of a trained set with its moments
        {"name": "densify_4m", "kind": "densify", "n": 4_000_000, "deg": 3},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(["step", "step", "step", "view", "autograd", "render", "serve", "ssim", "crossings", "init",
                       "densify"])
    c = {"kind": kind, "deg": rng.choice([0, 1, 2, 3, 3])}
    if kind == "ssim":
        c.update(views=_log(rng, 1, 16), w=_log(rng, 64, 2300), h=_log(rng, 64, 1800))
        del c["deg"]
        return c
    if kind == "crossings":
        del c["deg"]
        return dict(c, nx=_log(rng, 33, 512), ny=_log(rng, 33, 512), nz=_log(rng, 33, 512))
    c["scene"] = rng.choice(["gyroid", "blobs", "noise"])
    if kind == "init":
        return dict(c, n=_log(rng, 5_000, 4_000_000))
    if kind == "densify":
        del c["scene"]
        return dict(c, n=_log(rng, 5_000, 4_000_000))
    if kind == "autograd":
        return dict(c, scene="sphere", n=_log(rng, 2_000, 60_000), views=rng.randint(1, 4), w=_log(rng, 100, 900),
                    h=_log(rng, 100, 700))
    w, h = _log(rng, 200, 3840), _log(rng, 200, 2400)
    # a training batch or burst holds at most 64M pixels and 32M (view, Gaussian) pairs
    views = {"view": 1, "render": 1, "serve": rng.randint(3, 12)}.get(kind) or _log(rng, 1, 16)
    n = min(_log(rng, 20_000, 6_000_000), 32_000_000 // views)
    return dict(c, n=n, views=max(1, min(views, 64_000_000 // (w * h))), w=w, h=h)


# ---------------------------------------------------------------- inputs

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _field(scene, seed):
    if scene == "gyroid":
        phase = torch.rand(3, generator=_gen(seed), device=DEV, dtype=torch.float64) * 0.2
        return (lambda x: inputs._gyroid_fg(x + phase)), 0.0, 96
    if scene == "blobs":
        return inputs.BlobField(seed).fg, 0.5, 80
    return (lambda x: inputs._chunked(inputs.NoiseField(seed).fg, x, 1 << 21)), 0.0, 128


def _surface(scene, n, seed):
    """n points (float64) on a field's level set in contour-filter order, their unit normals and the point density
    per unit area."""
    g = _gen(seed)
    if scene == "sphere":
        x = torch.randn(n, 3, generator=g, device=DEV, dtype=torch.float64)
        x = x / x.norm(dim=1, keepdim=True)
        return x, x, n / (4 * math.pi)
    fg, iso, res = _field(scene, seed)
    half = SCENES[scene][1]
    h = 2 * half / res
    ax = torch.linspace(-half, half, res + 1, device=DEV, dtype=torch.float64)
    grid = torch.stack(torch.meshgrid(ax, ax, ax, indexing="ij"), -1).reshape(-1, 3)
    s = (fg(grid)[0] >= iso).view(res + 1, res + 1, res + 1)
    c = sum(s[i:res + i, j:res + j, k:res + k].int() for i in (0, 1) for j in (0, 1) for k in (0, 1))
    cells = torch.nonzero((c > 0) & (c < 8))
    got, normals, have = [], [], 0
    while have < n:
        m = int((n - have) * 1.15) + 64
        pick = cells[torch.randint(0, cells.shape[0], (m,), generator=g, device=DEV)]
        x0 = -half + h * (pick + torch.rand(m, 3, generator=g, device=DEV, dtype=torch.float64))
        x = x0
        for _ in range(2):  # Newton steps from a point of a cell that the level crosses
            f, d = fg(x)
            x = x - ((f - iso) / (d * d).sum(1).clamp_min(1e-30))[:, None] * d
        ok = ((x - x0).norm(dim=1) < 2 * h) & (x.abs() <= half).all(1) & (d.norm(dim=1) > 1e-12)
        got.append(x[ok])
        normals.append(d[ok] / d[ok].norm(dim=1, keepdim=True))
        have += int(got[-1].shape[0])
    x, nrm = torch.cat(got)[:n], torch.cat(normals)[:n]
    cell = ((x + half) / h).long().clamp_(0, res - 1)
    order = torch.argsort((cell[:, 2] * res + cell[:, 1]) * res + cell[:, 0], stable=True)
    # a plane of random direction crosses 1.5 cells per cell face of area
    return x[order], -nrm[order] if scene == "blobs" else nrm[order], n / (cells.shape[0] * h * h / 1.5)


def _scene(case, seed, perturbed):
    """Parameter planes [P, stride]: one flat Gaussian per surface point, sized by its three nearest neighbours'
    distances (drawn from their distribution at this density), Lambertian colour."""
    n, deg = case["n"], case["deg"]
    g = _gen(seed + 1)
    x, nrm, density = _surface(case["scene"], n, seed)
    p = torch.zeros(11 + 3 * (deg + 1) ** 2, inputs.padded_stride(n), device=DEV)
    p[0:3, :n] = x.t()
    e = torch.empty(3, n, device=DEV).exponential_(1.0, generator=g)
    ls = 0.5 * torch.log((3 * e[0] + 2 * e[1] + e[2]) / (3 * math.pi * density))
    if case["kind"] == "autograd":  # few, large splats of all shapes
        p[3:6, :n] = ls + 0.4 * torch.randn(3, n, generator=g, device=DEV)
        p[6:10, :n] = torch.randn(4, n, generator=g, device=DEV)
        p[10, :n] = 4 * torch.rand(n, generator=g, device=DEV) - 1
    else:
        p[3:6, :n] = ls
        p[5, :n] += math.log(0.3)
        w = 1 + nrm[:, 2]
        q = torch.stack([w, -nrm[:, 1], nrm[:, 0], torch.zeros_like(w)])
        q[:, w < 1e-6] = torch.tensor([0.0, 1.0, 0.0, 0.0], device=DEV, dtype=torch.float64)[:, None]
        p[6:10, :n] = q / q.norm(dim=0)
        p[10, :n] = 2.0
    light = (nrm.sum(1) / math.sqrt(3.0)).clamp_min(0.0)
    p[11:14, :n] = ((0.9 * light + 0.1 - 0.5) * 2 * math.sqrt(math.pi)).float()
    if deg:
        p[14:, :n] = 0.02 * torch.randn(p.shape[0] - 14, n, generator=g, device=DEV)
    if perturbed:  # 5 % off the reference set in every parameter
        u = 2 * torch.rand(p.shape, generator=g, device=DEV) - 1
        p = torch.where(p != 0, p * (1 + 0.05 * u), 0.05 * u)
    p[:, n:] = 0
    return p.contiguous()


def _cameras(case, seed):
    rng = random.Random(seed)
    radius, _ = SCENES[case["scene"]]
    w, h, kind = case["w"], case["h"], case["kind"]
    if kind == "view":
        radius *= 0.45
    cams = []
    for v in range(case["views"]):
        el = math.radians(rng.uniform(-75, 75))
        az = 2 * math.pi * rng.random()
        eye = [radius * math.cos(el) * math.cos(az), radius * math.cos(el) * math.sin(az), radius * math.sin(el)]
        s = {"serve": (1.0, 0.5, 0.25, 0.75), "autograd": (1.0, 0.61, 0.37)}.get(kind, (1.0,))
        s = s[v % len(s)]
        bg = (0.2, 0.5, 0.1) if kind == "autograd" else (0.0, 0.0, 0.0)
        cams.append(inputs.pinhole(inputs.look_at(eye), max(16, int(w * s)), max(16, int(h * s)), bg=bg))
    return cams


def _picture(cams, g):
    """Smooth images in [0, 1] in the batch layout, with a little noise."""
    out = []
    for c in cams:
        low = torch.rand(1, 3, 12, 16, generator=g, device=DEV)
        t = torch.nn.functional.interpolate(low, size=(c["height"], c["width"]), mode="bilinear")
        out.append(t.reshape(-1))
    t = torch.cat(out)
    return t.add_(0.02 * torch.rand(t.shape, generator=g, device=DEV)).clamp_(0, 1)


def _moments(p, n, pixels, g):
    """Adam moments as training leaves them: per plane of the size of this loss's gradients."""
    s = torch.empty_like(p).log_normal_(0.0, 1.0, generator=g) * (0.1 / pixels)
    m = torch.randn(p.shape, generator=g, device=DEV) * s * 0.3
    s[:, n:] = 0
    m[:, n:] = 0
    return m, s * s


def _volume(case, seed):
    """A volume whose values vary with the seed and whose side of the level 0.1 at a vertex does not, so that the
    number of crossings is the case's."""
    g = _gen(11)
    f = 0
    for n, axis in ((case["nz"], 0), (case["ny"], 1), (case["nx"], 2)):
        shape = [1, 1, 1]
        shape[axis] = n
        t = torch.linspace(0, 4 * math.pi, n, device=DEV) + torch.rand(1, generator=g, device=DEV)
        f = f + [torch.sin(t), torch.cos(1.3 * t), torch.sin(0.7 * t)][axis].view(shape)

    def smooth(g):
        low = torch.rand(1, 1, 24, 24, 24, generator=g, device=DEV)
        return torch.nn.functional.interpolate(low, size=f.shape, mode="trilinear")[0, 0]

    f = f + 0.5 * smooth(g) - 0.35
    f = torch.where(f.abs() < 1e-5, 1e-5, f)
    return (0.1 + f * (0.5 + smooth(_gen(seed)))).contiguous()


def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind, "case": case}
    g = _gen(seed + 2)
    if kind == "crossings":
        s.update(ctx=gs.Context(0), volume=_volume(case, seed))
        return s
    if kind == "ssim":
        cams = [inputs.pinhole(inputs.look_at((0.0, -3.0, 0.5)), case["w"], case["h"])] * case["views"]
        x = _picture(cams, g)
        y = (x + 0.1 * torch.randn(x.shape, generator=g, device=DEV)).clamp_(0, 1)
        ctx = gs.Context(0)
        tiny = inputs.sphere_scene(64, seed=1)  # the loss takes the view sizes of the batch last projected
        ctx.gs_project(torch.from_numpy(tiny["params"]).to(DEV), 64, 0, cams)
        s.update(ctx=ctx, x=x, y=y, loss=torch.zeros(1, device=DEV), grad=torch.empty_like(x))
        return s
    n, deg = case["n"], case["deg"]
    if kind == "densify":
        p = torch.zeros(11 + 3 * (deg + 1) ** 2, inputs.padded_stride(n), device=DEV)
        p[:, :n] = 0.3 * torch.randn(p.shape[0], n, generator=g, device=DEV)
        p[3:6, :n] -= 4.6
        p[10, :n] = 2.5 * p[10, :n] / 0.3
        m, v = _moments(p, n, 1e6, g)
        grad = 2e-4 * torch.empty(n, device=DEV).log_normal_(-0.8, 0.8, generator=g)
        count = torch.randint(0, 17, (n,), generator=g, device=DEV).float()
        # no decision within rounding of its threshold
        grad = torch.where((grad / 2e-4 - 1).abs() < 1e-4, 1e-4, grad) * count
        op, sz = torch.sigmoid(p[10].double()), p[3:6].amax(0).double().exp()
        p[10] = torch.where((op / 0.005 - 1).abs() < 1e-4, 1.0, p[10])
        p[3:6] = torch.where((sz / 0.01 - 1).abs() < 1e-4, p[3:6] - 0.01, p[3:6])
        p[:, n:] = 0
        cap = inputs.padded_stride(2 * n)
        outs = [torch.zeros(p.shape[0], cap, device=DEV) for _ in range(3)]
        s.update(ctx=gs.Context(0), p=p, m=m, v=v, grad=grad, count=count, outs=outs,
                 noise=torch.randn(n, 2, 3, generator=g, device=DEV))
        return s
    if kind == "init":
        m = n + n // 8
        x, nrm, _ = _surface(case["scene"], m, seed)
        sel = torch.sort(torch.randperm(m, generator=g, device=DEV)[:n])[0]
        out = torch.zeros(11 + 3 * (deg + 1) ** 2, inputs.padded_stride(n), device=DEV)
        s.update(ctx=gs.Context(0), points=x.float().contiguous(), normals=nrm.float().contiguous(), sel=sel, out=out)
        return s
    p = _scene(case, seed, perturbed=kind in ("step", "view"))
    cams = _cameras(case, seed)
    _, total = gs.image_offsets(cams)
    s.update(p=p, cams=cams)
    if kind == "serve":
        px = max(c["width"] * c["height"] for c in cams)
        s["srv"] = gs.Server(p, n, deg, slots=2, max_batch_views=8, memory_budget_bytes=12 << 30,
                             output_pool_bytes=0, max_view_pixels=px)
        s["outs"] = [torch.empty(3, c["height"], c["width"], device=DEV) for c in cams]
        torch.cuda.synchronize()  # the server's streams read the set from now on
        return s
    if kind == "render":
        s.update(ctx=gs.Context(0), image=torch.empty(total, device=DEV))
        return s
    if kind == "autograd":
        s.update(ctx=gs.Context(0), dimage=torch.randn(total, generator=g, device=DEV) / total)
        s["p"].requires_grad_(True)
        return s
    m, v = _moments(p, n, total, g)
    s.update(m=m, v=v, g=torch.zeros_like(p), target=_picture(cams, g), image=torch.empty(total, device=DEV),
             dimage=torch.empty(total, device=DEV), loss=torch.zeros(1, device=DEV), step=STEP0)
    if kind == "view":
        s["ctx"] = gs.Context(0)
        return s
    count = gs.Context(0)  # one uncaptured pass says how many tile instances the batch has
    count.gs_project(p, n, deg, cams)
    count.gs_bin_sort()
    inst = count.gs_get_counts()[0]
    count.close()
    ctx = gs.Context(0, instance_capacity=inst + inst // 4 + 65536)
    ctx.gs_train_graph_capture(s["p"], s["g"], m, v, n, deg, HP, cams, s["target"], s["image"], s["dimage"], s["loss"])
    s["ctx"] = ctx
    return s


# ---------------------------------------------------------------- one pass

def run(s):
    kind, case = s["kind"], s["case"]
    if kind == "step":
        s["step"] += 1
        s["ctx"].gs_train_graph_launch(s["cams"], s["target"], s["step"])
        return {k: s[k] for k in ("loss", "image", "g", "p", "m", "v")}
    if kind == "view":
        s["step"] += 1
        ctx, n, deg = s["ctx"], case["n"], case["deg"]
        ctx.gs_project(s["p"], n, deg, s["cams"])
        ctx.gs_bin_sort()
        ctx.gs_raster_fwd(s["image"])
        ctx.gs_ssim_loss(s["image"], s["target"], 0.2, s["loss"], s["dimage"])
        ctx.gs_raster_bwd(s["p"], n, deg, s["dimage"], s["g"])
        ctx.gs_adam(s["p"], s["g"], s["m"], s["v"], n, deg, dict(HP, visible_only=True), s["step"])
        return {k: s[k] for k in ("loss", "image", "g", "p", "m", "v")}
    if kind == "autograd":
        img = autograd.rasterize(s["p"], case["n"], case["deg"], s["cams"], s["ctx"])
        (grad,) = torch.autograd.grad(img, s["p"], s["dimage"])
        return {"image": img, "g": grad}
    if kind == "render":
        s["ctx"].gs_project(s["p"], case["n"], case["deg"], s["cams"])
        s["ctx"].gs_bin_sort()
        s["ctx"].gs_raster_fwd(s["image"])
        return {"image": s["image"]}
    if kind == "serve":
        tickets = [s["srv"].gs_serve_submit(c, out=o) for c, o in zip(s["cams"], s["outs"])]
        for t in tickets:
            status, _ = s["srv"].gs_serve_poll(t)
            if status != gs.GS_OK:
                raise RuntimeError("request %d: status %d" % (t, status))
            s["srv"].gs_serve_release(t)
        return s["outs"]
    if kind == "ssim":
        s["ctx"].gs_ssim_loss(s["x"], s["y"], 0.2, s["loss"], s["grad"])
        return {"loss": s["loss"], "grad": s["grad"]}
    if kind == "crossings":
        points, normals = s["ctx"].gs_iso_crossings(s["volume"], 0.1, (-1.0, -1.0, -1.0), (0.01, 0.01, 0.01))
        return {"points": points, "normals": normals}
    if kind == "init":
        s["ctx"].gs_init_gaussians(s["points"], s["normals"], s["out"], case["n"], case["deg"], select=s["sel"])
        return {"means": s["out"][:3], "scales": s["out"][3:6], "rest": s["out"][6:]}
    nout = s["ctx"].gs_densify(s["p"], s["m"], s["v"], case["n"], case["deg"], s["grad"], s["count"], s["noise"],
                               {"scene_extent": 1.0}, *s["outs"])
    return {"n": nout, "p": s["outs"][0], "m": s["outs"][1], "v": s["outs"][2]}


# ---------------------------------------------------------------- work

def work(case):
    """Bytes: inputs and outputs once.  Operations of the compositing: a pixel of these opaque surfaces takes about
    8 contributions before it stops, over about half of the image."""
    kind = case["kind"]
    if kind == "crossings":
        verts = case["nx"] * case["ny"] * case["nz"]
        points = 0.9 * verts ** (2.0 / 3.0) * 12  # about a dozen faces of the box of level surface
        return {"bytes": 4.0 * verts + 24.0 * points, "flops": 3.0 * verts + 100.0 * points}
    if kind == "ssim":
        count = 3.0 * case["views"] * case["w"] * case["h"]
        return {"bytes": 12.0 * count, "flops": count * (2 * 22 * 8 + 40)}
    n, planes = float(case["n"]), 11 + 3 * (case["deg"] + 1) ** 2
    if kind == "init":
        return {"bytes": n * (24 + 8 + 4 * planes), "flops": n * 40 * 9}
    if kind == "densify":
        return {"bytes": n * (2 * 3 * 4 * planes + 8 + 24), "flops": n * 40}
    pixels = 0.0
    for c in _cameras(case, 0):
        pixels += c["width"] * c["height"]
    pairs = n * case["views"]
    if kind in ("render", "serve"):
        return {"bytes": 4 * planes * n + 12 * pixels, "flops": pairs * (150 + 6 * (planes - 11)) + 4 * pixels * 19}
    flops = pairs * 3 * (150 + 6 * (planes - 11)) + 4 * pixels * 59
    if kind == "autograd":
        return {"bytes": 2 * 4 * planes * n + 24 * pixels, "flops": flops}
    # parameters, moments: read and written; gradients written; targets read, images and their gradients written
    return {"bytes": 7 * 4 * planes * n + 36 * pixels, "flops": flops + 12 * planes * n}


# ---------------------------------------------------------------- 64-bit restatement

def _sh_basis(d, deg):
    x, y, z = d.unbind(0)
    c = [torch.full_like(x, 0.5 / math.sqrt(math.pi))]
    if deg >= 1:
        a = math.sqrt(3 / (4 * math.pi))
        c += [a * y, a * z, a * x]
    if deg >= 2:
        a = 0.5 * math.sqrt(15 / math.pi)
        c += [a * x * y, a * y * z, 0.25 * math.sqrt(5 / math.pi) * (3 * z * z - 1), a * x * z,
              0.5 * a * (x * x - y * y)]
    if deg >= 3:
        e, f = 0.25 * math.sqrt(35 / (2 * math.pi)), 0.5 * math.sqrt(105 / math.pi)
        k = 0.25 * math.sqrt(21 / (2 * math.pi))
        c += [e * y * (3 * x * x - y * y), f * x * y * z, k * y * (5 * z * z - 1),
              0.25 * math.sqrt(7 / math.pi) * z * (5 * z * z - 3), k * x * (5 * z * z - 1),
              0.5 * f * z * (x * x - y * y), e * x * (x * x - 3 * y * y)]
    return torch.stack(c)


def _project64(p, deg, cam):
    """Rows mu_x, mu_y, A, B, C, opacity, r, g, b of each Gaussian; its tile rect and its FP32 depth."""
    vm = torch.tensor(cam["viewmat"], device=DEV, dtype=torch.float64)
    R, tau = vm[:3, :3], vm[:3, 3]
    mu = p[0:3]
    t = R @ mu + tau[:, None]
    r32, m32 = R.float(), mu.detach().float()
    depth = ((r32[2, 0] * m32[0] + r32[2, 1] * m32[1]) + r32[2, 2] * m32[2]) + tau[2].float()
    front = depth > cam["znear"]
    tz = torch.where(front, t[2], 1.0)
    W, H, fx, fy = cam["width"], cam["height"], cam["fx"], cam["fy"]
    mx, my = fx * t[0] / tz + cam["cx"], fy * t[1] / tz + cam["cy"]
    lx, ly = 1.3 * W / (2 * fx), 1.3 * H / (2 * fy)
    sx, sy = (t[0] / tz).clamp(-lx, lx), (t[1] / tz).clamp(-ly, ly)
    w, x, y, z = (p[6:10] / p[6:10].norm(dim=0)).unbind(0)
    rot = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                       2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                       2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)]).view(3, 3, -1)
    M = torch.einsum("ij,jkn->ikn", R, rot) * torch.exp(p[3:6])[None]
    u, v = fx / tz * (M[0] - sx * M[2]), fy / tz * (M[1] - sy * M[2])
    a, b, c = (u * u).sum(0) + 0.3, (u * v).sum(0), (v * v).sum(0) + 0.3
    det = a * c - b * b
    with torch.no_grad():
        lam = 0.5 * (a + c) + ((0.25 * (a - c) ** 2 + b * b).clamp_min(0.1)).sqrt()
        rad = torch.ceil(3 * lam.sqrt())
        gw, gh = (W + 15) // 16, (H + 15) // 16
        rect = [((q.detach() + s) / 16).floor().clamp(0, e).long()
                for q, s, e in ((mx, -rad, gw), (mx, rad + 15, gw), (my, -rad, gh), (my, rad + 15, gh))]
    eye = -R.t() @ tau
    d = mu - eye[:, None]
    Y = _sh_basis(d / d.norm(dim=0), deg)
    rgb = torch.stack([(Y * p[11 + ch::3]).sum(0) + 0.5 for ch in range(3)]).clamp_min(0.0)
    return torch.cat([torch.stack([mx, my, c / det, -b / det, a / det, torch.sigmoid(p[10])]), rgb]), rect, depth, front


def _tile_lists(rect, depth, front, gw):
    """Sorted (tile, depth, index) lists: the Gaussians, and per touched tile its first entry and length."""
    x0, x1, y0, y1 = rect
    count = ((x1 - x0).clamp_min(0) * (y1 - y0).clamp_min(0)) * front
    vis = torch.nonzero(count > 0)[:, 0]
    vis = vis[torch.argsort(depth[vis], stable=True)]
    k = count[vis]
    who = torch.repeat_interleave(vis, k)
    j = torch.arange(who.numel(), device=DEV) - torch.repeat_interleave(k.cumsum(0) - k, k)
    width = (x1 - x0)[who]
    tile = (y0[who] + j // width) * gw + x0[who] + j % width
    tile, order = torch.sort(tile, stable=True)
    tiles, length = torch.unique_consecutive(tile, return_counts=True)
    return who[order], tiles, length.cumsum(0) - length, length


def _composite64(q, cam, lists, image=None, dimage=None):
    """Writes the view's colours into image [3, H, W], or, with dimage, back-propagates them into q's gradient."""
    who, tiles, first, length = lists
    W, H = cam["width"], cam["height"]
    gw = (W + 15) // 16
    bg = torch.tensor(cam["bg"], device=DEV, dtype=torch.float64)
    at = torch.arange(256, device=DEV)
    order = torch.argsort(length)
    i, lens = 0, length[order].tolist()
    while i < len(lens):
        j, budget = i, 24_000_000 if dimage is not None else 80_000_000
        while j < len(lens) and (j + 1 - i) * lens[j] * 256 <= budget:
            j += 1
        j = max(j, i + 1)
        t = order[i:j]
        k = torch.arange(lens[j - 1], device=DEV)
        inside = k[None] < length[t][:, None]
        idx = who[(first[t][:, None] + k[None]).clamp_max(who.numel() - 1)]
        e = q[:, idx][..., None]  # [9, tiles, entries, 1]
        px = ((tiles[t] % gw) * 16)[:, None] + at % 16
        py = ((tiles[t] // gw) * 16)[:, None] + at // 16
        dx, dy = e[0] - px[:, None], e[1] - py[:, None]
        power = -0.5 * (e[2] * dx * dx + e[4] * dy * dy) - e[3] * dx * dy
        alpha = (e[5] * torch.exp(power)).clamp_max(0.99)
        with torch.no_grad():
            on = (power <= 0) & (alpha >= 1.0 / 255.0) & inside[..., None]
            on &= torch.cumprod(torch.where(on, 1 - alpha, 1.0), 1) >= 1e-4
        alpha = torch.where(on, alpha, 0.0)
        T = torch.exp(torch.cumsum(torch.log1p(-alpha), 1))
        wgt = alpha * torch.cat([torch.ones_like(T[:, :1]), T[:, :-1]], 1)
        C = torch.stack([(wgt * e[6 + ch]).sum(1) + T[:, -1] * bg[ch] for ch in range(3)])
        ok = (px < W) & (py < H)
        if dimage is None:
            image[:, py[ok], px[ok]] = C[:, ok]
        else:
            (C[:, ok] * dimage[:, py[ok], px[ok]]).sum().backward()
        i = j


def _views(flat, cams):
    sizes = [3 * c["width"] * c["height"] for c in cams]
    return [x.view(3, c["height"], c["width"]) for x, c in zip(flat.split(sizes), cams)]


def _render64(p, deg, cams):
    out = []
    with torch.no_grad():
        for cam in cams:
            q, rect, depth, front = _project64(p, deg, cam)
            img = torch.tensor(cam["bg"], device=DEV, dtype=torch.float64)[:, None, None].repeat(
                1, cam["height"], cam["width"])
            _composite64(q, cam, _tile_lists(rect, depth, front, (cam["width"] + 15) // 16), image=img)
            out.append(img)
    return out


def _grad64(p, deg, cams, dimages):
    """dL/dp, and which Gaussians' rects meet a view."""
    p = p.clone().requires_grad_(True)
    seen = torch.zeros(p.shape[1], dtype=torch.bool, device=DEV)
    for cam, dimg in zip(cams, dimages):
        q, rect, depth, front = _project64(p, deg, cam)
        seen |= front & (rect[1] > rect[0]) & (rect[3] > rect[2])
        leaf = q.detach().requires_grad_(True)
        _composite64(leaf, cam, _tile_lists(rect, depth, front, (cam["width"] + 15) // 16), dimage=dimg)
        q.backward(leaf.grad)
    return p.grad, seen


def _adam64(s, n, g, seen):
    lr = torch.full((g.shape[0], 1), HP["lr_sh_rest"], device=DEV, dtype=torch.float64)
    for rows, key in ((slice(0, 3), "mean"), (slice(3, 6), "scale"), (slice(6, 10), "quat"), (slice(10, 11), "opacity"),
                      (slice(11, 14), "sh_dc")):
        lr[rows] = HP["lr_" + key]
    b1, b2, t = HP["beta1"], HP["beta2"], STEP0 + 1
    p, m, v = (s[k].double() for k in "pmv")
    m1, v1 = b1 * m + (1 - b1) * g, b2 * v + (1 - b2) * g * g
    p1 = p - lr / (1 - b1 ** t) * m1 / (torch.sqrt(v1 / (1 - b2 ** t)) + HP["eps"])
    live = torch.zeros(p.shape[1], dtype=torch.bool, device=DEV)
    live[:n] = seen
    return [torch.where(live, a, b) for a, b in ((p1, p), (m1, m), (v1, v))]


def _blur(x):
    k = torch.arange(-5, 6, device=DEV, dtype=torch.float64)
    k = torch.exp(-k * k / 4.5)
    k = (k / k.sum()).tolist()
    h, w = x.shape[-2:]
    y = torch.nn.functional.pad(x, (0, 0, 5, 5))
    x = sum(k[i] * y[..., i:i + h, :] for i in range(11))
    y = torch.nn.functional.pad(x, (5, 5))
    return sum(k[i] * y[..., i:i + w] for i in range(11))


def _ssim_loss64(xs, ys, lam):
    """0.8 L1 + 0.2 (1 - SSIM) and its gradient, over lists of [3, H, W] images."""
    count = sum(x.numel() for x in xs)
    loss, grads = 0.0, []
    for x, y in zip(xs, ys):
        mx, my = _blur(x), _blur(y)
        sxx, syy, sxy = _blur(x * x) - mx * mx, _blur(y * y) - my * my, _blur(x * y) - mx * my
        n1, n2 = 2 * mx * my + 1e-4, 2 * sxy + 9e-4
        d1, d2 = mx * mx + my * my + 1e-4, sxx + syy + 9e-4
        ssim = n1 * n2 / (d1 * d2)
        dmx = 2 * my * (n2 - n1) / (d1 * d2) - ssim * 2 * mx * (1 / d1 - 1 / d2)
        ds = _blur(dmx) + 2 * x * _blur(-ssim / d2) + y * _blur(2 * n1 / (d1 * d2))
        loss = loss + ((1 - lam) * (x - y).abs().sum() + lam * (1 - ssim).sum()) / count
        grads.append(((1 - lam) * torch.sign(x - y) - lam * ds) / count)
    return loss.reshape(1), grads


def _nearest64(x):
    """Mean squared distance to the three nearest other points."""
    out = []
    for i in range(0, x.shape[0], 512):
        d = ((x[i:i + 512, None] - x[None]) ** 2).sum(-1)
        out.append(torch.topk(d, 4, dim=1, largest=False)[0][:, 1:].mean(1))
    return torch.cat(out)


def _exact_crossings(vol):
    f, iso = vol.double(), float(torch.tensor(0.1))
    h = float(torch.tensor(0.01))
    grads = []
    for axis in (2, 1, 0):
        g = torch.zeros_like(f)
        k = f.shape[axis]
        if k > 1:
            i = torch.arange(k, device=DEV)
            hi, lo = (i + 1).clamp_max(k - 1), (i - 1).clamp_min(0)
            shape = [1, 1, 1]
            shape[axis] = k
            g = (f.index_select(axis, hi) - f.index_select(axis, lo)) / ((hi - lo) * h).view(shape)
        grads.append(g)
    grad = torch.stack(grads, -1).view(-1, 3)
    nz, ny, nx = f.shape
    side, f = vol >= iso, f.view(-1)
    found = []
    for d, axis in enumerate((2, 1, 0)):
        k = f.new_zeros(0) if side.shape[axis] < 2 else side.narrow(axis, 0, side.shape[axis] - 1) != side.narrow(
            axis, 1, side.shape[axis] - 1)
        z, y, x = torch.nonzero(k, as_tuple=True)
        found.append(((z * ny + y) * nx + x) * 3 + d)
    e = torch.sort(torch.cat(found))[0]
    vert, d = e // 3, e % 3
    other = vert + torch.tensor([1, nx, nx * ny], device=DEV)[d]
    t = (iso - f[vert]) / (f[other] - f[vert])
    xyz = torch.stack([vert % nx, (vert // nx) % ny, vert // (nx * ny)], 1).double()
    xyz += t[:, None] * torch.nn.functional.one_hot(d, 3)
    n = grad[vert] + t[:, None] * (grad[other] - grad[vert])
    return {"points": -1.0 + h * xyz, "normals": n / n.norm(dim=1, keepdim=True)}


def _exact_densify(s, case):
    n, p = case["n"], s["p"].double()
    avg = torch.where(s["count"] > 0, s["grad"].double() / s["count"].clamp_min(1), 0.0)
    size = p[3:6, :n].amax(0).exp()
    kept = torch.sigmoid(p[10, :n]) >= 0.005
    grow = kept & (avg >= 2e-4)
    split = grow & (size > 0.01)
    reps = kept.long() + grow.long()
    src = torch.repeat_interleave(torch.arange(n, device=DEV), reps)
    k = torch.arange(src.numel(), device=DEV) - torch.repeat_interleave(reps.cumsum(0) - reps, reps)
    outs = [x.double()[:, src] for x in (s["p"], s["m"], s["v"])]
    fresh = split[src] | (k > 0)
    outs[1][:, fresh] = 0
    outs[2][:, fresh] = 0
    at = split[src]
    w, x, y, z = (p[6:10] / p[6:10].norm(dim=0))[:, src[at]].unbind(0)
    rot = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                       2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                       2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)]).view(3, 3, -1)
    step = outs[0][3:6, at].exp() * s["noise"].double()[src[at], k[at]].t()
    outs[0][0:3, at] += (rot * step[None]).sum(1)
    outs[0][3:6, at] -= math.log(0.8 * 2)
    pad = s["outs"][0].shape[1] - src.numel()
    p1, m1, v1 = (torch.nn.functional.pad(o, (0, pad)) for o in outs)
    return {"n": None, "p": p1, "m": m1, "v": v1}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("step", "view", "autograd") and case["n"] * case["views"] > 4_500_000:
        return None
    if kind in ("crossings", "ssim", "densify", "init"):
        s = prepare(case, seed)
        if kind == "crossings":
            return _exact_crossings(s["volume"])
        if kind == "densify":
            return _exact_densify(s, case)
        if kind == "ssim":
            shape = (case["views"], 3, case["h"], case["w"])
            loss, grads = _ssim_loss64([a.double() for a in s["x"].view(shape)], [a.double() for a in s["y"].view(shape)],
                                       0.2)
            return {"loss": loss, "grad": torch.cat([a.reshape(-1) for a in grads])}
        x, nrm = s["points"].double()[s["sel"]], s["normals"].double()[s["sel"]]
        w = 1 + nrm[:, 2]
        q = torch.stack([w, -nrm[:, 1], nrm[:, 0], torch.zeros_like(w)])
        q[:, w < 1e-6] = torch.tensor([0.0, 1.0, 0.0, 0.0], device=DEV, dtype=torch.float64)[:, None]
        rest = torch.zeros(s["out"].shape[0] - 6, s["out"].shape[1], device=DEV, dtype=torch.float64)
        rest[0:4, :case["n"]] = q / q.norm(dim=0)
        rest[4, :case["n"]] = 2.0
        rest[5:8, :case["n"]] = (0.9 * (nrm.sum(1) / math.sqrt(3.0)).clamp_min(0.0) - 0.4) * 2 * math.sqrt(math.pi)
        means = torch.zeros(3, s["out"].shape[1], device=DEV, dtype=torch.float64)
        means[:, :case["n"]] = x.t()
        scales = None
        if case["n"] <= 150_000:
            scales = torch.zeros_like(means)
            scales[:, :case["n"]] = 0.5 * torch.log(_nearest64(x).clamp_min(1e-14))
            scales[2, :case["n"]] += math.log(0.3)
        return {"means": means, "scales": scales, "rest": rest}
    n, deg = case["n"], case["deg"]
    cams = _cameras(case, seed)
    g = _gen(seed + 2)
    p32 = _scene(case, seed, perturbed=kind in ("step", "view"))
    p = p32.double()[:, :n].contiguous()
    images = _render64(p, deg, cams)
    flat = torch.cat([i.reshape(-1) for i in images])
    if kind == "serve":
        return images
    if kind == "render":
        return {"image": flat}
    if kind == "autograd":
        d32 = torch.randn(flat.numel(), generator=g, device=DEV) / flat.numel()
        grad, _ = _grad64(p, deg, cams, _views(d32.double(), cams))
        return {"image": flat, "g": torch.nn.functional.pad(grad, (0, p32.shape[1] - n))}
    m, v = _moments(p32, n, flat.numel(), g)
    target = _views(_picture(cams, g).double(), cams)
    if kind == "view":
        loss, dimages = _ssim_loss64(images, target, 0.2)
    else:
        loss = sum((a - b).abs().sum() for a, b in zip(images, target)).reshape(1) / flat.numel()
        dimages = [torch.sign(a - b) / flat.numel() for a, b in zip(images, target)]
    grad, seen = _grad64(p, deg, cams, dimages)
    if kind == "step":
        seen = torch.ones_like(seen)
    grad = torch.nn.functional.pad(grad, (0, p32.shape[1] - n))
    p1, m1, v1 = _adam64({"p": p32, "m": m, "v": v}, n, grad, seen)
    return {"loss": loss, "image": flat, "g": grad, "p": p1, "m": m1, "v": v1}
