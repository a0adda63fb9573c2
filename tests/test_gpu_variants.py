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


def test_crossings_emitted_into_too_small_outputs():
    """gs_iso_emit with a capacity below the count: the first crossings, nothing past them, GS_ECAPACITY by gs_sync."""
    import ctypes
    rng = np.random.default_rng(2)
    vol = torch.from_numpy(rng.uniform(-1.0, 1.0, (33, 40, 70)).astype(np.float32)).cuda()
    nz, ny, nx = vol.shape
    ctx = gs.Context(0)
    pts, nrm = ctx.gs_iso_crossings(vol, 0.1, (0.0, 0.0, 0.0), (1.0, 1.0, 1.0))
    m = pts.shape[0]
    work = torch.empty(ctx.L.gs_iso_workspace_bytes(nx, ny, nz), device="cuda", dtype=torch.uint8)
    zero, one = (ctypes.c_float * 3)(0, 0, 0), (ctypes.c_float * 3)(1, 1, 1)
    count = ctypes.c_int64()
    v, w = ctypes.c_void_p(vol.data_ptr()), ctypes.c_void_p(work.data_ptr())
    for cap in (0, 1, m // 2, m - 1, m):
        p = torch.full((m, 3), float("nan"), device="cuda")
        q = torch.full((m, 3), float("nan"), device="cuda")
        assert ctx.L.gs_iso_count(ctx.h, v, nx, ny, nz, ctypes.c_float(0.1), w, ctypes.byref(count)) == gs.GS_OK
        assert count.value == m
        assert ctx.L.gs_iso_emit(ctx.h, v, nx, ny, nz, ctypes.c_float(0.1), zero, one, w, ctypes.c_void_p(p.data_ptr()),
                                 ctypes.c_void_p(q.data_ptr()), cap) == gs.GS_OK
        if cap < m:
            with pytest.raises(gs.GsError):
                ctx.gs_sync()
        else:
            ctx.gs_sync()
        assert torch.equal(p[:cap], pts[:cap]) and torch.equal(q[:cap], nrm[:cap])
        assert torch.isnan(p[cap:]).all() and torch.isnan(q[cap:]).all()
    ctx.gs_sync()
    ctx.close()


def test_captured_step_of_many_tiles():
    """The automatic variants and tile order of a batch of many tiles, captured, against the one-pixel kernels in bin
    order call by call."""
    scene = inputs.random_scene(20000, 1, 21, extent=0.9, log_scale=(-6.0, -3.0))
    start = inputs.perturb(scene, 3)
    cams = [inputs.pinhole(inputs.look_at((0.4 + v, -2.8, 1.0)), w, h)
            for v, (w, h) in enumerate([(1511, 903), (640, 480)])]
    n, deg = start["n"], start["deg"]
    _, total = gs.image_offsets(cams)
    plain = gs.Context(0)
    for opt, val in ((gs.GS_OPT_RASTER_FWD, 1), (gs.GS_OPT_RASTER_BWD, 1), (gs.GS_OPT_TILE_ORDER, 0)):
        plain.gs_set_option(opt, val)
    _, target = run_forward(plain, scene, cams)
    inst = plain.gs_get_counts()[0]
    hp = dict(lr_mean=1e-3, lr_scale=5e-3, lr_quat=1e-3, lr_opacity=0.05, lr_sh_dc=2.5e-3, lr_sh_rest=1e-4)
    p = torch.from_numpy(start["params"]).cuda()
    g, m, v = (torch.zeros_like(p) for _ in range(3))
    img, d, loss = torch.empty(total, device="cuda"), torch.empty(total, device="cuda"), torch.zeros(1, device="cuda")
    ctx = gs.Context(0, instance_capacity=2 * inst + 65536)
    ctx.gs_train_graph_capture(p, g, m, v, n, deg, hp, cams, target, img, d, loss)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert sum(((c["width"] + 15) // 16) * ((c["height"] + 15) // 16) for c in cams) >= 32 * sms
    assert [ctx.gs_get_option(o) for o in (gs.GS_OPT_RASTER_FWD, gs.GS_OPT_RASTER_BWD, gs.GS_OPT_TILE_ORDER)] == [4, 8, 1]
    ctx.gs_train_graph_launch(cams, target, 1)
    ctx.gs_sync()
    q, ref = run_forward(plain, start, cams)
    assert (img - ref).abs().max().item() <= 1e-6
    # (dL/dimage from the captured step's image, so that no sign of image - target differs)
    grads = torch.full_like(q, float("nan"))
    plain.gs_raster_bwd(q, n, deg, d, grads)
    plain.gs_sync()
    a, b = (t.cpu().numpy().astype(np.float64) for t in (g, grads))
    assert rel_l2(a, b) <= 2e-5
    assert torch.isfinite(p).all()
    ctx.close()
    plain.close()
