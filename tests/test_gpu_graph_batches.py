"""A captured training step whose context takes other work between replays
(GPU only): each replay leaves the captured batch as the context's current
one, in workspaces of its own, whatever came before it."""
import numpy as np
import pytest
import torch

from paper_2509_05216_gb300 import gs, inputs
from tests.gpu_helpers import expected_binning, run_forward
from tests.test_gpu_graph import HP, State, render, setup

pytestmark = pytest.mark.gpu


def smaller(ctx, scene):
    """One small view, projected and binned only."""
    ctx.gs_project(torch.from_numpy(scene["params"]).cuda(), scene["n"], scene["deg"],
                   [inputs.pinhole(inputs.look_at((0.4, -2.8, 1.0)), 64, 48)])
    ctx.gs_bin_sort()


def larger(ctx, scene):
    """More and larger views than captured: the workspaces grow."""
    run_forward(ctx, scene, [inputs.pinhole(inputs.look_at((0.4 + v, -2.8, 1.0)), 400, 300) for v in range(5)])


def points(ctx, scene):
    """Initial Gaussians of a point cloud larger than the set (shares the sort's workspaces)."""
    pts = torch.rand(200000, 3, device="cuda")
    out = torch.zeros((14, 200000), device="cuda")
    ctx.gs_init_gaussians(pts, torch.nn.functional.normalize(pts, dim=1), out, 200000, 0)


@pytest.mark.parametrize("between", [[smaller], [larger], [points], [larger, smaller], [smaller, larger, points]])
def test_replays_keep_the_captured_batch(between):
    ref, cur, cams = setup()
    n, deg = cur["n"], cur["deg"]
    plain = gs.Context(0)
    targets = render(plain, ref, cams)
    inst, _, _ = plain.gs_get_counts()
    _, total = gs.image_offsets(cams)
    tiles = sum(((c["width"] + 15) // 16) * ((c["height"] + 15) // 16) for c in cams)
    runs = []
    for disturbed in (False, True):
        st = State(cur)
        img, d, loss = torch.empty(total, device="cuda"), torch.empty(total, device="cuda"), torch.zeros(1, device="cuda")
        ctx = gs.Context(0, instance_capacity=32 * inst + 65536)
        ctx.gs_train_graph_capture(st.p, st.g, st.m, st.v, n, deg, HP, cams, targets, img, d, loss)
        losses = []
        for step in range(1, 4):
            if disturbed:
                for work in between:
                    work(ctx, ref)
            p0 = st.p.clone()
            ctx.gs_train_graph_launch(cams, targets, step)
            ctx.gs_sync()
            losses.append(loss.item())
            if step == 1:
                first = img.clone()
            if not disturbed:
                continue
            got, bins, pixels = ctx.gs_get_counts()
            assert bins == tiles and pixels * 3 == total
            rec = [ctx.gs_get_buffer(b).cpu().numpy() for b in (gs.GS_BUF_REC0, gs.GS_BUF_REC2, gs.GS_BUF_REC3)]
            keys, vals, ranges, _ = expected_binning(*rec, cams, n, st.p.shape[1])
            assert got == keys.size
            assert np.array_equal(ctx.gs_get_buffer(gs.GS_BUF_RANGES).cpu().numpy().astype(np.int64), ranges)
            assert np.array_equal(ctx.gs_get_buffer(gs.GS_BUF_VALS).cpu().numpy().astype(np.int64), vals)
            # the replay's own backward again, from the context's state
            again = torch.full_like(st.g, float("nan"))
            ctx.gs_raster_bwd(p0, n, deg, d, again)
            ctx.gs_sync()
            assert (torch.linalg.norm(again - st.g) / torch.linalg.norm(st.g)).item() <= 1e-4
        runs.append((first, losses))
        ctx.close()
    assert torch.equal(runs[0][0], runs[1][0])
    for a, b in zip(runs[0][1], runs[1][1]):
        assert abs(a - b) <= 1e-4 * a
    plain.close()


def test_a_larger_set_is_captured_anew():
    """Capture, outgrow the workspaces, capture a larger set: the second graph trains the second set."""
    ref, cur, cams = setup()
    big = inputs.random_scene(30000, 1, 7, extent=0.7)
    plain = gs.Context(0)
    targets = render(plain, big, cams)
    inst, _, _ = plain.gs_get_counts()
    _, total = gs.image_offsets(cams)
    img, d, loss = torch.empty(total, device="cuda"), torch.empty(total, device="cuda"), torch.zeros(1, device="cuda")
    ctx = gs.Context(0, instance_capacity=32 * inst + 65536)
    for scene in (cur, big):
        st = State(scene)
        ctx.gs_train_graph_capture(st.p, st.g, st.m, st.v, scene["n"], scene["deg"], HP, cams, targets, img, d, loss)
        ctx.gs_train_graph_launch(cams, targets, 1)
        ctx.gs_sync()
        larger(ctx, ref)
    # (the last replay rendered `big`, whose own render are the targets)
    ctx.gs_train_graph_launch(cams, targets, 2)
    ctx.gs_sync()
    assert torch.isfinite(st.p).all() and loss.item() <= 0.2
    ctx.close()
    plain.close()


def test_an_impossible_request_leaves_the_graph():
    """A workspace that no memory could hold is refused (GS_ENOMEM), and the captured step goes on."""
    ref, cur, cams = setup()
    n, deg = cur["n"], cur["deg"]
    plain = gs.Context(0)
    targets = render(plain, ref, cams)
    inst, _, _ = plain.gs_get_counts()
    _, total = gs.image_offsets(cams)
    images = []
    for disturbed in (False, True):
        st = State(cur)
        img, d, loss = torch.empty(total, device="cuda"), torch.empty(total, device="cuda"), torch.zeros(1, device="cuda")
        ctx = gs.Context(0, instance_capacity=2 * inst + 1024)
        ctx.gs_train_graph_capture(st.p, st.g, st.m, st.v, n, deg, HP, cams, targets, img, d, loss)
        if disturbed:
            # 64 views of 65,536^2 projected (no pixel buffer is touched); the image loss's partials would take 9 TB
            huge = [inputs.pinhole(inputs.look_at((0.4, -2.8, 1.0)), 65536, 65536)] * 64
            ctx.gs_project(torch.from_numpy(ref["params"]).cuda(), n, deg, huge)
            with pytest.raises(gs.GsError, match="cudaMalloc"):
                ctx.gs_ssim_loss(img, targets, 0.2, loss, d)
        ctx.gs_train_graph_launch(cams, targets, 1)
        ctx.gs_sync()
        images.append(img.clone())
        ctx.close()
    assert torch.equal(images[0], images[1])
    plain.close()
