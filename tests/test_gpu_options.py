"""Options that follow the batch until set, and again once set to automatic
(GPU only)."""
import math

import pytest
import torch

from paper_2509_05216_gb300 import gs, inputs
from tests.gpu_helpers import run_forward

pytestmark = pytest.mark.gpu

AUTOMATIC = (gs.GS_OPT_RASTER_FWD, gs.GS_OPT_RASTER_BWD, gs.GS_OPT_TILE_ORDER)


def test_automatic_options_come_back():
    scene = inputs.random_scene(500, 0, 3, extent=0.5)
    few = [inputs.pinhole(inputs.look_at((0.4, -2.8, 1.0)), 100, 80)]
    many = [inputs.pinhole(inputs.look_at((0.4, -2.8, 1.0)), 2048, 2048)]  # 16,384 tiles, 100 per SM
    ctx = gs.Context(0)
    assert [ctx.gs_get_option(o) for o in AUTOMATIC] == [2, 4, 0]  # (nothing projected yet)

    def read(cams):
        _, img = run_forward(ctx, scene, cams)
        return [ctx.gs_get_option(o) for o in AUTOMATIC], img

    small, image = read(few)
    large, _ = read(many)
    assert small == [2, 4, 0] and large == [4, 8, 1]
    for opt, value in zip(AUTOMATIC, (8, 1, 0)):
        ctx.gs_set_option(opt, value)
    assert read(few)[0] == [8, 1, 0] and read(many)[0] == [8, 1, 0]
    for opt in AUTOMATIC:
        ctx.gs_set_option(opt, gs.GS_OPT_AUTO)
    again, img = read(few)
    assert again == small and torch.equal(img, image) and read(many)[0] == large
    for opt in (gs.GS_OPT_BWD_DIRECT, gs.GS_OPT_SORT_ITEMS, gs.GS_OPT_SORT_WAIT):
        with pytest.raises(gs.GsError):
            ctx.gs_set_option(opt, gs.GS_OPT_AUTO)
    with pytest.raises(gs.GsError):
        ctx.gs_set_option(gs.GS_OPT_RASTER_FWD, 0)
    with pytest.raises(gs.GsError):
        ctx.gs_set_option(gs.GS_OPT_TILE_ORDER, -2)
    ctx.close()


def test_many_tiles_of_long_lists():
    """Many tiles with 2,048 pairs each or more: list order, but the kernels of fewer pixels per thread."""
    cams = [inputs.pinhole(inputs.look_at((2.8 * math.cos(0.1 * v), 2.8 * math.sin(0.1 * v), 0.5)), 208, 96) for v in range(63)]
    for n, kernels in ((159000, (4, 8, 1)), (161000, (2, 4, 1))):  # 63 n / 4,914 tiles: 2,038 and 2,064
        scene = inputs.random_scene(n, 0, 4, extent=0.8, log_scale=(-6.5, -5.5))
        ctx = gs.Context(0)
        _, img = run_forward(ctx, scene, cams)
        got = tuple(ctx.gs_get_option(o) for o in AUTOMATIC)
        if torch.cuda.get_device_properties(0).multi_processor_count == 152:
            assert got == kernels
        for opt, value in zip(AUTOMATIC, (1, 1, 0)):
            ctx.gs_set_option(opt, value)
        assert (run_forward(ctx, scene, cams)[1] - img).abs().max().item() <= 1e-6
        ctx.close()


# (tiles per SM, pairs per tile) on both sides of the lines between the backward kernels; 152 SMs; tall views count as
# 2.3 focal lengths (30 tiles of 500), wide ones whole
@pytest.mark.parametrize("w,h,n,kernel", [(192, 192, 23039, 4), (192, 192, 23040, 1), (208, 192, 25000, 2), (208, 192, 160000, 1),
                                          (400, 384, 98000, 2), (416, 384, 110000, 4), (2048, 2048, 30000, 8),
                                          (240, 8000, 30000, 4), (8000, 240, 30000, 8), (240, 8000, 90000, 2)])
def test_backward_kernel_by_tiles_and_pairs(w, h, n, kernel):
    scene = inputs.random_scene(n, 0, 4, extent=0.8, log_scale=(-6.0, -5.0))
    cams = [inputs.pinhole(inputs.look_at((0.4, -2.8, 1.0)), w, h)]
    ctx = gs.Context(0)
    p, img = run_forward(ctx, scene, cams)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    if sms == 152:
        assert ctx.gs_get_option(gs.GS_OPT_RASTER_BWD) == kernel
    dimg = torch.randn(img.shape, generator=torch.Generator(device="cuda").manual_seed(1), device="cuda")
    grads = [torch.full_like(p, float("nan")) for _ in range(2)]
    ctx.gs_raster_bwd(p, n, 0, dimg, grads[0])
    ctx.gs_set_option(gs.GS_OPT_RASTER_BWD, 4)
    ctx.gs_raster_bwd(p, n, 0, dimg, grads[1])
    ctx.gs_sync()
    a, b = (g[:, :n].double() for g in grads)
    assert torch.isfinite(a).all() and ((a - b).norm() / b.norm()).item() <= 2e-5
    ctx.close()
