"""Densification of small and large sets, whose passes take one or four
Gaussians per thread and fewer or more planes per block (GPU only), against
the oracle."""
import numpy as np
import pytest
import torch

from oracle import densify as OD
from paper_2509_05216_gb300 import gs

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


# blocks of 256: one short, full, one over; several; either side of 5 blocks of 1,024 per SM (152 SMs)
@pytest.mark.parametrize("n,deg", [(255, 0), (256, 3), (257, 2), (30001, 3), (778239, 0), (778241, 0)])
def test_densify_sizes(n, deg):
    rng = np.random.default_rng(n)
    stride = n + (-n) % 4
    P = 11 + 3 * (deg + 1) ** 2
    p = rng.normal(size=(P, stride)).astype(np.float32)
    p[3:6] = rng.uniform(-6.0, -3.0, (3, stride))
    p[10] = rng.uniform(-7.0, 3.0, stride)
    m, v = (rng.normal(size=(P, stride)).astype(np.float32) for _ in range(2))
    # (nothing within rounding of a threshold: gradients away from 2e-4, sizes and opacities away from theirs)
    avg = np.where(rng.uniform(size=n) < 0.6, rng.uniform(3e-4, 1e-3, n), rng.uniform(0.0, 1e-4, n))
    cnt = rng.integers(0, 5, n).astype(np.float32)
    grad = (avg * cnt).astype(np.float32)
    size, op = np.exp(p[3:6].astype(np.float64)).max(0), 1 / (1 + np.exp(-p[10].astype(np.float64)))
    p[3:6, np.abs(size / 0.02 - 1) < 1e-4] -= 0.01
    p[10, np.abs(op / 0.005 - 1) < 1e-4] += 0.01
    noise = rng.normal(size=(n, 2, 3)).astype(np.float32)
    f64 = [a.astype(np.float64) for a in (p[:, :n], m[:, :n], v[:, :n], grad, cnt, noise)]
    rp, rm, rv, _ = OD.densify(*f64, tau=2e-4, dense=0.01, extent=2.0, min_opacity=0.005, split_n=2)
    outs = [torch.full((P, 2 * stride), float("nan"), device="cuda") for _ in range(3)]
    ctx = gs.Context(0)
    nout = ctx.gs_densify(dev(p), dev(m), dev(v), n, deg, dev(grad), dev(cnt), dev(noise), dict(scene_extent=2.0), *outs)
    ctx.gs_sync()
    assert nout == rp.shape[1]
    po, mo, vo = (o[:, :nout].cpu().numpy() for o in outs)
    # a split sample's mean: three products of FP32 factors (exp to 2 ulp) up to about 0.05 * 5 beside a mean of up to 5
    np.testing.assert_allclose(po.astype(np.float64), rp, rtol=1e-6, atol=2e-6)
    np.testing.assert_array_equal(mo.astype(np.float64), rm)
    np.testing.assert_array_equal(vo.astype(np.float64), rv)
    assert all(bool(torch.isnan(o[:, nout:]).all()) for o in outs)
    ctx.close()
