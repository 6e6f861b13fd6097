"""Histograms with larger stencils at the edges of the tiled kernel's range:
row bounds (8 | 9, 16 | 17 bins), one type alone, tiles' remainders in x, y
and z, point masses, against the oracle."""
import numpy as np
import pytest
import torch

import helpers as H_

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ucp():
    from paper_2407_18015_gb300 import build
    build.build()
    from paper_2407_18015_gb300 import ucp as u
    return u


@pytest.mark.parametrize("bins", [1, 8, 9, 16, 17])
@pytest.mark.parametrize("stencil,shape", [(1, (1, 9, 33)), (2, (1, 17, 70)), (2, (1, 1, 40)),
                                           (3, (3, 5, 33)), (3, (1, 6, 40)), (3, (4, 8, 32))])
def test_stencil_histogram_tiles(ucp, orc, bins, stencil, shape):
    D, H, W = shape
    rng = np.random.default_rng(bins * 10 + stencil + W)
    p = H_.random_params(2, D * H, W, rng, bins=bins)
    pm = rng.random((D * H, W)) < 0.15
    p[1][pm] = p[0][pm]
    p = p.astype(np.float32).reshape((2 + bins,) + ((D, H, W) if D > 1 else (H, W)))
    dev = torch.from_numpy(p).cuda()
    ctx = ucp.Context(0)
    for boundary in (0, 1):
        desc = ucp.make_desc("histogram", bins=bins, stencil=stencil, depth=D, boundary=boundary)
        pmin, pmax, st = ctx.probability_from_params(dev, desc)
        only_min = ctx.probability_from_params(dev, desc, ucp.UCP_MIN)[0]
        only_max = ctx.probability_from_params(dev, desc, ucp.UCP_MAX)[1]
        torch.cuda.synchronize()
        assert torch.equal(only_min, pmin) and torch.equal(only_max, pmax)
        rmin, rmax, rst = orc.prob_stencil(p.astype(np.float64), 2, stencil, bins=bins,
                                           boundary=boundary)
        assert np.abs(pmin.cpu().numpy().reshape(rmin.shape) - rmin).max() <= 1e-5
        assert np.abs(pmax.cpu().numpy().reshape(rmax.shape) - rmax).max() <= 1e-5
        np.testing.assert_array_equal(st.cpu().numpy().reshape(rst.shape), rst)
