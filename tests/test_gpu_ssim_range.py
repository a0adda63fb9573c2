"""SSIM far outside [0, 1], where the denominators of its map leave the range
whose reciprocal is a normal FP32 number: quotients, against the FP64 oracle
(GPU only)."""
import numpy as np
import pytest
import torch

from oracle import ssim as OS
from paper_2509_05216_gb300 import gs, inputs

pytestmark = pytest.mark.gpu


# (scale, second image).  Two equal images of uniform values in [0.5, 1] scale: the map's denominator
# (mx^2 + my^2 + C1)(sxx + syy + C2) is 0.05 scale^4 in the middle and at most 0.23 scale^4 at the border (by the
# oracle's window sums), so at 6e9 it stays finite and crosses 2^126, above which its reciprocal is subnormal.
# Beside a black image, at 1e11, it is infinite, and the map 0.
@pytest.mark.parametrize("scale,second", [(1.0, "equal"), (6e9, "equal"), (1e-12, "equal"), (1e11, "black"),
                                          (1e11, "black first")])
def test_ssim_of_large_and_small_values(scale, second):
    w, h = 75, 67
    cams = [inputs.pinhole(inputs.look_at((0.4, -2.8, 1.0)), w, h)]
    scene = inputs.random_scene(64, 0, 3, extent=0.5)
    ctx = gs.Context(0)
    ctx.gs_project(torch.from_numpy(scene["params"]).cuda(), scene["n"], scene["deg"], cams)
    rng = np.random.default_rng(4)
    x = (scale * rng.uniform(0.5, 1.0, (3, h, w))).astype(np.float32)
    y = x if second == "equal" else np.zeros_like(x)
    if second == "black first":
        x, y = y, x
    dx, dy = (torch.from_numpy(np.ascontiguousarray(a)).cuda().reshape(-1) for a in (x, y))
    ssim, psnr = ctx.gs_image_metrics(dx, dy, 1)
    # a quotient of two products of FP32 sums: a few dozen roundings of 6e-8, and the differences E[x^2] - mx^2
    # (0.04 of their terms) on both sides of an equal pair alike
    assert abs(ssim[0] - OS.ssim(x, y)) <= 1e-5
    if second != "equal":
        assert abs(psnr[0] - OS.psnr(x, y)) <= 1e-4
    loss, grad = torch.zeros(1, device="cuda"), torch.full_like(dx, float("nan"))
    ctx.gs_ssim_loss(dx, dy, 0.2, loss, grad)
    ctx.gs_sync()
    ref, _ = OS.dssim_loss([x], [y], 0.2)
    assert abs(loss.item() - ref) <= 1e-5 * max(1.0, abs(ref))
    assert torch.isfinite(grad).all()
    ctx.close()


# One-pixel views: the window sums are the pixel's value times the centre weight twice, so the map follows from a few
# FP32 operations.  The quotient is by one reciprocal and a Newton step for denominators of ordinary images and by
# division beyond; both are within an ulp of the IEEE quotient.
@pytest.mark.parametrize("scale", [1e-3, 1.0, 40.0, 3e3, 1e5])
def test_ssim_map_is_the_ieee_quotient(scale):
    views = 64
    cams = [inputs.pinhole(inputs.look_at((0.4, -2.8, 1.0)), 1, 1)] * views
    scene = inputs.random_scene(64, 0, 3, extent=0.5)
    ctx = gs.Context(0)
    ctx.gs_project(torch.from_numpy(scene["params"]).cuda(), scene["n"], scene["deg"], cams)
    f, wide = np.float32, np.longdouble
    win = np.exp(-((np.arange(11) - 5.0) ** 2) / 4.5)
    w5, c1, c2, two = f(win[5] / win.sum()), f(0.01) * f(0.01), f(0.03) * f(0.03), f(2)

    def fma(a, b, c):
        return (wide(a) * b.astype(wide) + wide(c)).astype(f)

    def window(a):
        return w5 * (w5 * a)

    for seed in range(8):
        rng = np.random.default_rng(seed)
        x, y = (f(scale) * rng.uniform(0, 1, views).astype(f) for _ in range(2))
        mx, my = window(x), window(y)
        sxx, syy, sxy = fma(-mx, mx, window(x * x)), fma(-my, my, window(y * y)), fma(-mx, my, window(x * y))
        n1, n2 = fma(two * mx, my, c1), fma(two, sxy, c2)
        d1, d2 = fma(mx, mx, my * my) + c1, sxx + syy + c2
        ref = n1 * n2 / (d1 * d2)
        assert ref.dtype == f
        dx, dy = (torch.from_numpy(np.repeat(a, 3)).cuda() for a in (x, y))  # three equal channels
        got, _ = ctx.gs_image_metrics(dx, dy, views)
        assert np.all(np.abs(np.array(got) - ref) <= np.spacing(np.abs(ref)) * (1 + 1e-6))
    ctx.close()


# every number of rows per strip (4 to 128, by the batch's pixels) and both block sizes, with ragged last strips
@pytest.mark.parametrize("sizes", [[(61, 67)], [(301, 299)], [(515, 511)], [(701, 763)], [(1027, 1001)], [(1919, 1081)],
                                   [(1451, 1449), (1453, 1447)], [(97, 131)] * 5 + [(300, 20)]])
def test_strips_of_every_length(sizes):
    cams = [inputs.pinhole(inputs.look_at((0.4, -2.8, 1.0)), w, h) for w, h in sizes]
    scene = inputs.random_scene(64, 0, 3, extent=0.5)
    ctx = gs.Context(0)
    ctx.gs_project(torch.from_numpy(scene["params"]).cuda(), scene["n"], scene["deg"], cams)
    rng = np.random.default_rng(sizes[0][0])
    xs = [rng.uniform(0, 1, (3, h, w)).astype(np.float32) for w, h in sizes]
    ys = [np.clip(x + rng.normal(0, 0.1, x.shape), 0, 1).astype(np.float32) for x in xs]
    x, y = (torch.from_numpy(np.concatenate([a.reshape(-1) for a in v])).cuda() for v in (xs, ys))
    loss, grad = torch.zeros(1, device="cuda"), torch.full_like(x, float("nan"))
    for _ in range(2):  # (the second call finds the first one's state)
        ctx.gs_ssim_loss(x, y, 0.2, loss, grad)
    ctx.gs_sync()
    ref, ref_grads = OS.dssim_loss(xs, ys, 0.2)
    # the tolerances of the strips' small batches: FP32 window sums, means over thousands of pixels
    assert abs(loss.item() - ref) <= 1e-6
    for g, r in zip(gs.split_images(grad, cams), ref_grads):
        g = g.cpu().numpy().astype(np.float64)
        assert np.linalg.norm(g - r) <= 1e-5 * np.linalg.norm(r)
    ssim, psnr = ctx.gs_image_metrics(x, y, len(cams))
    for v in range(len(cams)):
        assert abs(ssim[v] - OS.ssim(xs[v], ys[v])) <= 2e-6 and abs(psnr[v] - OS.psnr(xs[v], ys[v])) <= 1e-4
    ctx.close()
