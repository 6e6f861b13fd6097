"""Epanechnikov pieces where factors never start on the centre's support:
neighbours up to 1e6 widths away (ramps), narrow beside wide supports, point
masses; minimum, maximum, saddle, larger stencils and gradient against the
oracle."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ucp():
    from paper_2407_18015_gb300 import build
    build.build()
    from paper_2407_18015_gb300 import ucp as u
    return u


def _params(ramp, seed):
    H, W = 11, 37
    rng = np.random.default_rng(seed)
    m = rng.normal(0, 0.5, (H, W)) + ramp * (np.arange(W)[None, :] % 5) * (np.arange(H)[:, None] % 3)
    w = 10.0 ** rng.uniform(-2, 0.3, (H, W))
    w[rng.random((H, W)) < 0.1] = 0.0
    return np.stack([m, w]).astype(np.float32)


@pytest.mark.parametrize("ramp", [0.0, 1.0, 3e2, 1e4])
def test_far_and_narrow_neighbours(ucp, orc, ramp):
    p = _params(ramp, seed=int(ramp) + 3)
    p64 = p.astype(np.float64)
    dev = torch.from_numpy(p).cuda()
    ctx = ucp.Context(0)
    desc = ucp.make_desc("epanechnikov")
    pmin, pmax, _ = ctx.probability_from_params(dev, desc)
    sad, _ = ctx.saddle_from_params(dev, desc)
    rmin, rmax, _ = orc.prob(p64, 1)
    rsad = orc.saddle(p64, 1)[0]
    for g, r in ((pmin, rmin), (pmax, rmax), (sad, rsad)):
        assert np.abs(g.cpu().numpy() - r).max() <= 1e-5
    for stencil in (1, 2):
        d = ucp.make_desc("epanechnikov", stencil=stencil)
        g = ctx.probability_from_params(dev, d)
        r = orc.prob_stencil(p64, 1, stencil)
        for a, b in zip(g[:2], r[:2]):
            assert np.abs(a.cpu().numpy() - b).max() <= 1e-5
    wt = np.random.default_rng(9).uniform(0, 1, p.shape[1:]).astype(np.float32)
    for cp in (1, 2):
        g = ctx.backward(dev, desc, cp, torch.from_numpy(wt).cuda()).cpu().numpy()
        r = orc.grad(p64, 1, wt.astype(np.float64), cptype=cp)
        assert (np.abs(g - r) <= 1e-4 * np.abs(r) + 2e-5 * max(1.0, np.abs(r).max())).all()
