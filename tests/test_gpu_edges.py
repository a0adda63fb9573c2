"""Kernels at the sizes where their partitions can go wrong, against the
oracles (GPU only): words, blocks and ragged rows of the crossings, blocks and
sample counts of the densification."""
import numpy as np
import pytest
import torch

from oracle import densify as OD
from oracle import init as OI
from paper_2509_05216_gb300 import gs, inputs

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
