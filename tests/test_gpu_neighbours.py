"""Neighbour scales of point sets whose box is long, flat or both, where the
finest grid takes more cells along the longer sides (GPU only), against the
oracle."""
import numpy as np
import pytest
import torch

from oracle import init as OI
from paper_2509_05216_gb300 import gs

pytestmark = pytest.mark.gpu

# sides of the box, in every order of the axes: a line, a thin one, a ribbon, a plane, a slab, a bar, a cube; the
# last two ends of the bits that a side takes (none; one cell less and one more than a power of two)
SIDES = [(1.0, 0.0, 0.0), (0.0, 1.0, 0.0), (1e-4, 0.0, 1.0), (0.01, 1.0, 0.0), (1.0, 1.0, 0.0), (0.0, 1.0, 1.0),
         (1.0, 0.05, 1.0), (0.02, 0.02, 1.0), (1.0, 1.0, 1.0), (1.0, 0.4999, 0.5001), (0.2501, 1.0, 0.2499)]


@pytest.mark.parametrize("sides", SIDES)
@pytest.mark.parametrize("n", [5, 3000, 60000])
def test_scales_of_long_and_flat_sets(sides, n):
    rng = np.random.default_rng(n + SIDES.index(sides))
    pts = rng.uniform(0.0, 1.0, (n, 3)) * np.array(sides)
    if n >= 3000:  # a dense part, and a few points that must look far
        pts[: n // 3] = pts[0] + (pts[: n // 3] - pts[0]) * 2e-3
    pts = (pts[rng.permutation(n)] * 3.0).astype(np.float32)
    out = torch.zeros((14, n + (-n) % 4), device="cuda")
    nrm = torch.zeros(n, 3, device="cuda")
    nrm[:, 2] = 1.0
    ctx = gs.Context(0)
    ctx.gs_init_gaussians(torch.from_numpy(pts).cuda(), nrm, out, n, 0)
    ctx.gs_sync()
    # FP32 differences of the coordinates are exact to 6e-8 of themselves, the sum of squares and the logarithm add a few roundings
    np.testing.assert_allclose(out[3, :n].cpu().numpy(), OI.knn_log_scales(pts), rtol=0, atol=2e-5)
    ctx.close()
