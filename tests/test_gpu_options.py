"""Options that follow the batch until set, and again once set to automatic
(GPU only)."""
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
