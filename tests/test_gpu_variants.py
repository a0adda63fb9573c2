"""Variants that smaller scenes do not reach (GPU only): the sort's partition
sizes on segments long enough to take them, the per-lane atomics of the
backward kernels that have them, single gradient elements across kernels."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2509_05216_gb300 import gs, inputs
from tests.gpu_helpers import expected_binning, rel_l2, run_forward, to_dev_images

pytestmark = pytest.mark.gpu


# segments of up to 262,144 keys take 4 or 8 keys per thread whatever is set
@pytest.mark.parametrize("items", [12, 16, 20, 24])
def test_sort_partition_sizes_of_long_segments(items):
    scene = inputs.random_scene(700000, 0, 5, extent=0.9, log_scale=(-6.0, -5.0))
    cams = [inputs.pinhole(inputs.look_at((0.4 + v, -2.8, 1.0)), 320 - 16 * v, 200) for v in range(2)]
    n, stride = scene["n"], scene["params"].shape[1]
    ctx = gs.Context(0)
    ctx.gs_set_option(gs.GS_OPT_SORT_ITEMS, items)
    run_forward(ctx, scene, cams)
    bufs = [ctx.gs_get_buffer(b).cpu().numpy() for b in (gs.GS_BUF_REC0, gs.GS_BUF_REC2, gs.GS_BUF_REC3)]
    keys, vals, ranges, per_view = expected_binning(*bufs, cams, n, stride)
    # (a segment's length is taken as the batch's room over the views: pairs for the depths, instances for the tiles)
    assert stride > 262144 and per_view.sum() > 2 * 262144
    assert np.array_equal(ctx.gs_get_buffer(gs.GS_BUF_KEYS).cpu().numpy().view(np.uint32),
                          (keys >> np.uint64(32)).astype(np.uint32))
    assert np.array_equal(ctx.gs_get_buffer(gs.GS_BUF_VALS).cpu().numpy().astype(np.int64), vals)
    assert np.array_equal(ctx.gs_get_buffer(gs.GS_BUF_RANGES).cpu().numpy().astype(np.int64), ranges)
    ctx.close()


def mixed():
    scene = inputs.random_scene(6000, 1, 12, extent=0.8)
    cams = [inputs.pinhole(inputs.look_at((0.4, -2.8, 1.0)), 160, 120, bg=(0.1, 0.2, 0.3)),
            inputs.pinhole(inputs.look_at((2.5, 1.0, -1.2)), 97, 131)]
    return scene, cams


@pytest.mark.parametrize("direct", [0, 3, 32])
@pytest.mark.parametrize("bwd", [1, 2])
def test_direct_atomics_match_oracle(bwd, direct):
    scene, cams = mixed()
    O.build()
    ctx = gs.Context(0)
    ctx.gs_set_option(gs.GS_OPT_RASTER_BWD, bwd)
    ctx.gs_set_option(gs.GS_OPT_BWD_DIRECT, direct)
    p, _ = run_forward(ctx, scene, cams)
    rng = np.random.default_rng(8)
    dimgs = [rng.normal(size=(3, c["height"], c["width"])) * (~O.render(scene, c)[2]) for c in cams]
    grads = torch.zeros_like(p)
    ctx.gs_raster_bwd(p, scene["n"], scene["deg"], to_dev_images(dimgs), grads)
    ctx.gs_sync()
    ref = O.render_grad(scene, cams, dimgs)
    n = scene["n"]
    keep = np.ones(n, bool)
    for cam in cams:
        keep &= (O.gaussian_flags(scene, cam) & O.G_MARG_ANY_GRAD) == 0
    g = grads.cpu().numpy().astype(np.float64)
    assert rel_l2(g[:, :n][:, keep], ref[:, :n][:, keep]) <= 1e-3
    ctx.close()


def test_backward_kernels_agree_in_every_element():
    """From one set of parameters and one dL/dimage, each gradient element of every backward kernel within 1e-4 of its
    plane's largest of the one-pixel kernel's: T is recovered over at most a few hundred contributors at 2^-22 each (7e-5), and the sums of
    different order add less."""
    scene, cams = mixed()
    _, total = gs.image_offsets(cams)
    dimg = torch.from_numpy(np.random.default_rng(3).normal(size=total).astype(np.float32)).cuda()
    out = {}
    for bwd in (1, 2, 4, 8):
        ctx = gs.Context(0)
        ctx.gs_set_option(gs.GS_OPT_RASTER_BWD, bwd)
        p, _ = run_forward(ctx, scene, cams)
        out[bwd] = torch.full_like(p, float("nan"))
        ctx.gs_raster_bwd(p, scene["n"], scene["deg"], dimg, out[bwd])
        ctx.gs_sync()
        ctx.close()
    largest = out[1].abs().amax(1, keepdim=True)
    for bwd in (2, 4, 8):
        assert torch.isfinite(out[bwd]).all()
        assert ((out[bwd] - out[1]).abs() / largest).max().item() <= 1e-4, bwd


# enough (view, Gaussian) pairs for the flags of those that took a gradient: one word of views, three with a last one
# that is not whole, all 64; ragged tiles
@pytest.mark.parametrize("n,views", [(1200001, 3), (200003, 18), (60001, 64)])
@pytest.mark.parametrize("bwd", [4, 8])
def test_backward_of_flagged_pairs(n, views, bwd):
    scene = inputs.random_scene(n, 0, 6, extent=0.8, log_scale=(-5.5, -4.0))
    cams = [inputs.pinhole(inputs.look_at((2.8 * np.cos(0.1 * v), 2.8 * np.sin(0.1 * v), 0.5)), 47 + v % 3, 50)
            for v in range(views)]
    assert n * views >= 3500000 and 4 * n * views >= 3 * sum(c["width"] * c["height"] for c in cams)
    _, total = gs.image_offsets(cams)
    dimg = torch.from_numpy(np.random.default_rng(7).normal(size=total).astype(np.float32)).cuda()
    out = {}
    for kernel in (1, bwd):  # (the one-pixel kernel keeps no flags)
        ctx = gs.Context(0)
        ctx.gs_set_option(gs.GS_OPT_RASTER_BWD, kernel)
        stat, count = torch.zeros(n, device="cuda"), torch.zeros(n, device="cuda")
        ctx.gs_set_densify_stats(stat, count)
        p, _ = run_forward(ctx, scene, cams)
        grads = torch.full_like(p, float("nan"))
        ctx.profile_reset()
        ctx.gs_raster_bwd(p, n, 0, dimg, grads)
        ctx.gs_sync()
        launched = {k["name"] for k in ctx.profile_read() if k["launches"]}
        assert ("pair_masks" in launched) == (kernel != 1)
        out[kernel] = [t.cpu().numpy().astype(np.float64) for t in (grads, stat, count)]
        ctx.gs_set_densify_stats(None, None)
        ctx.close()
    assert np.isfinite(out[bwd][0]).all() and rel_l2(out[bwd][0], out[1][0]) <= 2e-5
    assert rel_l2(out[bwd][1], out[1][1]) <= 2e-5 and np.array_equal(out[bwd][2], out[1][2])


def test_small_batches_keep_no_flags():
    """Below 3.5M pairs the flags' clear and launch cost more than they save, however few the pixels."""
    scene, _ = mixed()
    cams = [inputs.pinhole(inputs.look_at((0.4 + v, -2.8, 1.0)), 48, 32) for v in range(2)]
    _, total = gs.image_offsets(cams)
    ctx = gs.Context(0)
    p, _ = run_forward(ctx, scene, cams)
    ctx.profile_reset()
    ctx.gs_raster_bwd(p, scene["n"], scene["deg"], torch.ones(total, device="cuda"), torch.zeros_like(p))
    ctx.gs_sync()
    assert not any(k["name"] == "pair_masks" and k["launches"] for k in ctx.profile_read())
    ctx.close()
