"""Histogram supports down to one unit in the last place beside wide ones: the
edges of such a support round to a few positions of the centre's frame, where
its survival falls almost like a point mass's.  From parameters (minimum,
maximum, both at once, saddle) and fitted (one model, the fused models, the
batch), against the oracle."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
TOL = 1e-5


@pytest.fixture(scope="module")
def ucp():
    from paper_2407_18015_gb300 import build
    build.build()
    from paper_2407_18015_gb300 import ucp as u
    return u


def _up(H, W):
    y, x = np.mgrid[0:H, 0:W]
    return (y + x) % 2 == 0


def _params(H, W, bins, seed):
    """A checkerboard of wide supports and of ones of half width 1e-8 .. 1
    inside them, a quarter of these one unit in the last place wide; the
    narrow ones' masses in the first and the last bin."""
    rng = np.random.default_rng(seed)
    up = _up(H, W)
    c = np.where(up, rng.normal(0, 0.2, (H, W)), rng.uniform(-0.6, 0.6, (H, W)))
    hw = np.where(up, rng.uniform(0.5, 1, (H, W)), 10.0 ** rng.uniform(-8, 0, (H, W)))
    lo, hi = (c - hw).astype(np.float32), (c + hw).astype(np.float32)
    ulp = ~up & (rng.random((H, W)) < 0.25)
    hi[ulp] = np.nextafter(lo[ulp], np.float32(2))
    m = rng.uniform(0, 1, (bins, H, W))
    m[1:-1, ~up] *= 0.02
    m /= m.sum(axis=0, keepdims=True)
    return np.concatenate([np.stack([lo, hi]), m]).astype(np.float32)


@pytest.mark.parametrize("bins", [2, 5, 8, 16])
def test_from_params(ucp, orc, bins):
    p = _params(33, 70, bins, seed=bins)
    dev = torch.from_numpy(p).cuda()
    ctx = ucp.Context(0)
    desc = ucp.make_desc("histogram", bins=bins)
    pmin, pmax, _ = ctx.probability_from_params(dev, desc)
    only_min = ctx.probability_from_params(dev, desc, ucp.UCP_MIN)[0]
    only_max = ctx.probability_from_params(dev, desc, ucp.UCP_MAX)[1]
    sad, _ = ctx.saddle_from_params(dev, desc)
    p64 = p.astype(np.float64)
    rmin, rmax, _ = orc.prob(p64, 2, bins=bins)
    rsad = orc.saddle(p64, 2, bins=bins)[0]
    for got, ref, tol in ((pmin, rmin, TOL), (only_min, rmin, TOL), (pmax, rmax, TOL),
                          (only_max, rmax, TOL), (sad, rsad, 2 * TOL)):
        assert np.abs(got.cpu().numpy() - ref).max() <= tol


@pytest.mark.parametrize("bins", [5, 8, 16])
@pytest.mark.parametrize("W", [64, 63])
def test_fitted(ucp, orc, bins, W):
    """Members one unit in the last place apart at every other vertex."""
    H, N = 40, 20
    rng = np.random.default_rng(bins + W)
    ens = rng.normal(0, 0.5, (N, H, W)).astype(np.float32)
    flat = ~_up(H, W)
    a = rng.uniform(-0.6, 0.6, (H, W)).astype(np.float32)
    two = np.where(rng.random((N, H, W)) < 0.5, a, np.nextafter(a, np.float32(2)))
    ens[:, flat] = two[:, flat]
    dev = torch.from_numpy(ens).cuda()
    ctx = ucp.Context(0)
    desc = ucp.make_desc("histogram", bins=bins)
    p64 = ctx.fit(dev, desc).double().cpu().numpy()
    rmin, rmax, _ = orc.prob(p64, 2, bins=bins)
    rsad = orc.saddle(p64, 2, bins=bins)[0]
    got = [(r, g) for r, g in zip((rmin, rmax), ctx.probability(dev, desc)[:2])]
    got.append((rsad, ctx.saddle(dev, desc)[0]))
    descs = [ucp.make_desc("uniform"), ucp.make_desc("epanechnikov"), desc]
    out = [[torch.empty((H, W), device="cuda") for _ in descs] for _ in range(2)]
    ucp.ucp_probability_models(ctx.handle, dev, descs, 3, out[0], out[1])
    got += [(rmin, out[0][2]), (rmax, out[1][2])]
    batch = ucp.Batch(ctx)
    bmin, bmax = (torch.empty((H, W), device="cuda") for _ in range(2))
    batch.add(dev, desc, ucp.UCP_MIN, bmin, None)
    batch.add(dev, desc, ucp.UCP_MAX, None, bmax)
    batch.run()
    got += [(rmin, bmin), (rmax, bmax)]
    torch.cuda.synchronize()
    for ref, g in got:
        assert np.abs(g.cpu().numpy() - ref).max() <= (2 if ref is rsad else 1) * TOL
