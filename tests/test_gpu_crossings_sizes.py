"""Crossings of volumes on either side of the size from which a block takes
1,024 words instead of 64 (GPU only)."""
import numpy as np
import pytest

from paper_2509_05216_gb300 import gs
from tests.test_gpu_edges import dev, edge_points

pytestmark = pytest.mark.gpu


# 2^18 words are 8,388,608 vertices: one row less, one column more; ragged rows and planes in blocks of each size
@pytest.mark.parametrize("shape", [(1, 2896, 2896), (1, 2896, 2897), (7, 1101, 1103), (33, 257, 1001)])
def test_crossings_of_large_volumes(shape):
    z, y, x = np.meshgrid(*[np.arange(s, dtype=np.float64) for s in shape], indexing="ij", sparse=True)
    vol = (np.sin(0.11 * x + 0.05 * z) + np.cos(0.07 * y + 0.4 * z) + 0.1 * np.sin(0.9 * x * y / max(shape))).astype(np.float32)
    vol[np.abs(vol - 0.1) < 1e-3] = 0.3
    ctx = gs.Context(0)
    pts, nrm = ctx.gs_iso_crossings(dev(vol), 0.1, (0.0, 0.0, 0.0), (1.0, 1.0, 1.0))
    ref = edge_points(vol, 0.1)
    assert ref.shape[0] > 100000 and pts.shape[0] == ref.shape[0]
    # FP32: a coordinate's rounding (up to 2,897: 1.3e-4), t of values at least 1e-3 from the level
    np.testing.assert_allclose(pts.cpu().numpy(), ref, rtol=0, atol=4e-7 * max(shape) + 1e-4)
    assert np.abs(np.linalg.norm(nrm.cpu().numpy(), axis=1) - 1).max() <= 1e-5
    ctx.close()
