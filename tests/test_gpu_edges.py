"""Kernels at the sizes where their partitions can go wrong, against the
oracles (GPU only): words, blocks and ragged rows of the crossings, blocks and
sample counts of the densification, strips of the image loss, uneven point
sets, sort and emission partitions, tiles and pair flags of the compositing
backwards."""
import numpy as np
import pytest
import torch

from oracle import densify as OD
from oracle import init as OI
from oracle import ssim as OS
from paper_2509_05216_gb300 import gs, inputs
from tests.gpu_helpers import expected_binning, rel_l2, run_forward

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def edge_points(vol, iso):
    """Crossing points of a unit grid in vertex order (any axis may have one sample)."""
    f = vol.astype(np.float64)
    inside = vol >= np.float32(iso)
    rows = []
    for d, axis in enumerate((2, 1, 0)):
        lo = [slice(None)] * 3
        hi = [slice(None)] * 3
        lo[axis], hi[axis] = slice(0, -1), slice(1, None)
        z, y, x = np.nonzero(inside[tuple(lo)] != inside[tuple(hi)])
        a = f[z, y, x]
        b = f[z + (axis == 0), y + (axis == 1), x + (axis == 2)]
        p = np.stack([x, y, z], 1).astype(np.float64)
        p[:, d] += (np.float64(np.float32(iso)) - a) / (b - a)
        rows.append(np.concatenate([((z * vol.shape[1] + y) * vol.shape[2] + x)[:, None] * 3.0 + d, p], 1))
    r = np.concatenate(rows)
    return r[np.argsort(r[:, 0]), 1:]


# rows shorter than, equal to and longer than a 32-vertex word, words spanning rows and planes, single-sample
# axes, and more than one block of 32,768 vertices
@pytest.mark.parametrize("shape", [(1, 1, 1), (1, 1, 2), (1, 2, 1), (2, 1, 1), (1, 1, 70000), (3, 1, 31), (5, 32, 1),
                                   (2, 3, 5), (1, 9, 33), (4, 5, 32), (3, 7, 65), (9, 64, 64), (33, 31, 37),
                                   (2, 129, 255)])
def test_crossings_of_ragged_volumes(shape):
    rng = np.random.default_rng(sum(shape))
    vol = rng.uniform(-1.0, 1.0, shape).astype(np.float32)
    vol[np.abs(vol - 0.1) < 1e-3] = 0.3
    ctx = gs.Context(0)
    pts, nrm = ctx.gs_iso_crossings(dev(vol), 0.1, (0.0, 0.0, 0.0), (1.0, 1.0, 1.0))
    ref = edge_points(vol, 0.1)
    assert pts.shape[0] == ref.shape[0]
    # FP32: the interpolated coordinate is below max(shape), t carries a few roundings of the two differences
    np.testing.assert_allclose(pts.cpu().numpy(), ref, rtol=0, atol=4e-7 * max(shape) + 1e-6)
    if min(shape) >= 2 and max(shape) < 100:
        rp, rn = OI.iso_crossings(vol, float(np.float32(0.1)), (0.0, 0.0, 0.0), (1.0, 1.0, 1.0))
        np.testing.assert_allclose(ref, rp, rtol=0, atol=1e-9)
        cos = np.sum(nrm.cpu().numpy().astype(np.float64) * rn, axis=1)
        assert cos.min() > 1 - 1e-5
    ctx.close()


@pytest.mark.parametrize("n,split_n,opacity", [(1, 2, 2.0), (1023, 1, None), (1024, 3, None), (1025, 4, None),
                                               (2500, 2, -9.0), (2049, 2, None)])
def test_densify_blocks_and_sample_counts(n, split_n, opacity):
    rng = np.random.default_rng(n + split_n)
    deg, stride = 1, n + (-n) % 4
    P = 11 + 3 * (deg + 1) ** 2
    p = rng.normal(size=(P, stride)).astype(np.float32)
    p[3:6] = rng.uniform(-6.0, -3.0, (3, stride))
    p[10] = opacity if opacity is not None else rng.uniform(-7.0, 3.0, stride)
    m, v = (rng.normal(size=(P, stride)).astype(np.float32) for _ in range(2))
    avg = np.where(rng.uniform(size=n) < 0.6, rng.uniform(3e-4, 1e-3, n), rng.uniform(0.0, 1e-4, n))
    cnt = rng.integers(0, 5, n).astype(np.float32)
    grad = (avg * cnt).astype(np.float32)
    noise = rng.normal(size=(n, split_n, 3)).astype(np.float32)
    f64 = [a.astype(np.float64) for a in (p[:, :n], m[:, :n], v[:, :n], grad, cnt, noise)]
    rp, rm, rv, _ = OD.densify(*f64, tau=2e-4, dense=0.01, extent=2.0, min_opacity=0.005, split_n=split_n)
    outs = [torch.full((P, 4 * stride), float("nan"), device="cuda") for _ in range(3)]
    ctx = gs.Context(0)
    nout = ctx.gs_densify(dev(p), dev(m), dev(v), n, deg, dev(grad), dev(cnt), dev(noise),
                          dict(scene_extent=2.0, split_n=split_n), *outs)
    ctx.gs_sync()
    assert nout == rp.shape[1]
    po, mo, vo = (o[:, :nout].cpu().numpy().astype(np.float64) for o in outs)
    np.testing.assert_allclose(po, rp, rtol=1e-6, atol=2e-6)
    np.testing.assert_array_equal(mo, rm)
    np.testing.assert_array_equal(vo, rv)
    assert all(bool(torch.isnan(o[:, nout:]).all()) for o in outs)  # nothing past the outputs
    ctx.close()


# strips of 32 columns and 32 rows: narrower, exact, one more; a batch of ragged views
@pytest.mark.parametrize("sizes", [[(16, 16)], [(32, 32)], [(33, 31)], [(31, 65), (64, 20)], [(97, 129), (16, 200)]])
def test_ssim_strips(sizes):
    cams = [inputs.pinhole(inputs.look_at((0.4, -2.8, 1.0)), w, h) for w, h in sizes]
    scene = inputs.random_scene(64, 0, 3, extent=0.5)
    ctx = gs.Context(0)
    ctx.gs_project(dev(scene["params"]), scene["n"], scene["deg"], cams)
    rng = np.random.default_rng(len(sizes) + sizes[0][0])
    xs = [rng.uniform(0, 1, (3, h, w)).astype(np.float32) for w, h in sizes]
    ys = [np.clip(x + rng.normal(0, 0.1, x.shape), 0, 1).astype(np.float32) for x in xs]
    x, y = (dev(np.concatenate([a.reshape(-1) for a in v])) for v in (xs, ys))
    loss, grad = torch.zeros(1, device="cuda"), torch.full_like(x, float("nan"))
    ctx.gs_ssim_loss(x, y, 0.2, loss, grad)
    ctx.gs_sync()
    ref, ref_grads = OS.dssim_loss(xs, ys, 0.2)
    assert abs(loss.item() - ref) <= 1e-6
    for g, r in zip(gs.split_images(grad, cams), ref_grads):
        assert rel_l2(g.cpu().numpy().astype(np.float64), r) <= 1e-5
    ssim, psnr = ctx.gs_image_metrics(x, y, len(cams))
    for v in range(len(cams)):
        assert abs(ssim[v] - OS.ssim(xs[v], ys[v])) <= 2e-6 and abs(psnr[v] - OS.psnr(xs[v], ys[v])) <= 1e-4
    x[5] = float("inf")  # an infinite pixel makes the sums infinite or NaN, not finite
    ctx.gs_ssim_loss(x, y, 0.0, loss, None)
    _, psnr = ctx.gs_image_metrics(x, y, len(cams))
    assert not np.isfinite(loss.item()) and psnr[0] == -np.inf
    ctx.close()


@pytest.mark.parametrize("kind", ["four", "line", "grid", "cluster_outliers", "duplicates", "uniform"])
def test_neighbour_scales_of_uneven_sets(kind):
    rng = np.random.default_rng(17)
    if kind == "four":
        pts = rng.uniform(-1, 1, (4, 3))
    elif kind == "line":  # one axis only
        pts = np.stack([rng.uniform(-5, 5, 1025), np.zeros(1025), np.zeros(1025)], 1)
    elif kind == "grid":  # every distance tied, points on cell borders
        pts = np.stack(np.meshgrid(*[np.arange(16.0)] * 3), -1).reshape(-1, 3)
    elif kind == "cluster_outliers":  # a cluster in a few of the finest cells, and points that must look far
        pts = np.concatenate([rng.normal(0, 2e-3, (3000, 3)), rng.uniform(-1, 1, (40, 3)), [[1.0, 1.0, 1.0]]])
    elif kind == "duplicates":
        pts = np.repeat(rng.uniform(-1, 1, (700, 3)), 5, axis=0)
    else:
        pts = rng.uniform(0, 1, (40001, 3))
    pts = pts[rng.permutation(pts.shape[0])].astype(np.float32)
    n = pts.shape[0]
    nrm = np.tile(np.float32([0, 0, 1]), (n, 1))
    out = torch.zeros((14, n + (-n) % 4), device="cuda")
    ctx = gs.Context(0)
    ctx.gs_init_gaussians(dev(pts), dev(nrm), out, n, 0)
    ctx.gs_sync()
    ref = OI.knn_log_scales(pts)
    # FP32 differences of coordinates up to 5: 3e-7 absolute on each distance
    near = np.exp(ref)
    np.testing.assert_allclose(out[3, :n].cpu().numpy(), ref, rtol=0, atol=2e-5 + 6e-7 / near.min() * (kind != "duplicates"))
    ctx.close()


# segments on either side of the sizes at which the sorts and the emission change their keys per thread, one view
# (partitions in ticket order) and several
@pytest.mark.parametrize("n,views", [(255, 1), (1025, 3), (66000, 1), (66000, 2), (270001, 1), (700000, 2)])
def test_binning_sizes(n, views):
    scene = inputs.random_scene(n, 0, 5, extent=0.9, log_scale=(-6.0, -5.0))
    cams = [inputs.pinhole(inputs.look_at((0.4 + v, -2.8, 1.0)), 320 - 16 * v, 200) for v in range(views)]
    ctx = gs.Context(0)
    run_forward(ctx, scene, cams)
    bufs = [ctx.gs_get_buffer(b).cpu().numpy() for b in (gs.GS_BUF_REC0, gs.GS_BUF_REC2, gs.GS_BUF_REC3)]
    keys, vals, ranges, _ = expected_binning(*bufs, cams, n, scene["params"].shape[1])
    assert np.array_equal(ctx.gs_get_buffer(gs.GS_BUF_KEYS).cpu().numpy().view(np.uint32),
                          (keys >> np.uint64(32)).astype(np.uint32))
    assert np.array_equal(ctx.gs_get_buffer(gs.GS_BUF_VALS).cpu().numpy().astype(np.int64), vals)
    assert np.array_equal(ctx.gs_get_buffer(gs.GS_BUF_RANGES).cpu().numpy().astype(np.int64), ranges)
    ctx.close()


# 16 x 16 tiles cut by the image border, one pixel, an odd tile count; few pixels for the Gaussians (the pairs that
# take a gradient are flagged) and many
@pytest.mark.parametrize("n,sizes", [(40, [(16, 16)]), (3000, [(17, 15), (1, 1), (33, 47)]), (20000, [(64, 48), (50, 30)]),
                                     (500, [(320, 200), (100, 90)])])
def test_backward_variants_agree(n, sizes):
    scene = inputs.random_scene(n, 1, 9, extent=0.8)
    cams = [inputs.pinhole(inputs.look_at((0.4 + v, -2.8, 1.0)), w, h, bg=(0.1, 0.2, 0.3))
            for v, (w, h) in enumerate(sizes)]
    _, total = gs.image_offsets(cams)
    dimg = dev(np.random.default_rng(n).normal(size=total).astype(np.float32))
    ctx = gs.Context(0)
    out = {}
    for fwd, bwd in ((1, 1), (1, 4), (2, 2), (2, 4), (2, 8), (4, 4), (8, 8)):
        ctx.gs_set_option(gs.GS_OPT_RASTER_FWD, fwd)
        ctx.gs_set_option(gs.GS_OPT_RASTER_BWD, bwd)
        stat, count = torch.zeros(n, device="cuda"), torch.zeros(n, device="cuda")
        ctx.gs_set_densify_stats(stat, count)
        p, img = run_forward(ctx, scene, cams)
        grads = torch.full_like(p, float("nan"))
        for _ in range(2):  # a second backward of the same forward: the same gradients, the statistic again
            ctx.gs_raster_bwd(p, n, scene["deg"], dimg, grads)
        ctx.gs_sync()
        out[fwd, bwd] = [t.cpu().numpy().astype(np.float64) for t in (img, grads, stat, count)]
        ctx.gs_set_densify_stats(None, None)
    ref = out[1, 1]
    for key, got in out.items():
        assert np.abs(got[0] - ref[0]).max() <= 1e-6, key
        assert np.isfinite(got[1]).all() and rel_l2(got[1], ref[1]) <= 2e-5, key
        assert rel_l2(got[2], ref[2]) <= 2e-5 and np.array_equal(got[3], ref[3]), key
    ctx.close()


# enough tiles for the order of longest lists and the kernels of many tiles: several blocks of 1,024 tiles, ragged
def test_many_tiles_in_order():
    sizes = [(1111, 703), (640, 480), (1500, 900)]
    scene = inputs.random_scene(30000, 1, 21, extent=0.9, log_scale=(-6.0, -3.0))
    cams = [inputs.pinhole(inputs.look_at((0.4 + v, -2.8, 1.0)), w, h) for v, (w, h) in enumerate(sizes)]
    _, total = gs.image_offsets(cams)
    dimg = dev(np.random.default_rng(5).normal(size=total).astype(np.float32))
    tiles = sum(((w + 15) // 16) * ((h + 15) // 16) for w, h in sizes)
    out = []
    for plain in (True, False):
        ctx = gs.Context(0)
        if plain:
            for opt, val in ((gs.GS_OPT_RASTER_FWD, 1), (gs.GS_OPT_RASTER_BWD, 1), (gs.GS_OPT_TILE_ORDER, 0)):
                ctx.gs_set_option(opt, val)
        p, img = run_forward(ctx, scene, cams)
        grads = torch.full_like(p, float("nan"))
        ctx.gs_raster_bwd(p, scene["n"], scene["deg"], dimg, grads)
        ctx.gs_sync()
        if not plain and tiles >= 32 * torch.cuda.get_device_properties(0).multi_processor_count:
            assert ctx.gs_get_option(gs.GS_OPT_TILE_ORDER) == 1 and ctx.gs_get_option(gs.GS_OPT_RASTER_BWD) == 8
        out.append([t.cpu().numpy().astype(np.float64) for t in (img, grads)])
        ctx.close()
    assert np.abs(out[0][0] - out[1][0]).max() <= 1e-6
    assert np.isfinite(out[1][1]).all() and rel_l2(out[1][1], out[0][1]) <= 2e-5
