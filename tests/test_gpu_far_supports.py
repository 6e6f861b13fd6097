"""Histogram walks over supports near the end of the float range: a neighbour
that starts far below the centre's support (below -2e38 in its frame) must
not be walked past its last row.  Disjoint supports have exact answers; a
support that reaches into the centre's is compared with the oracle."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ucp():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2407_18015_gb300 import build
    build.build()
    from paper_2407_18015_gb300 import ucp as u
    return u


def _params(bins, low):
    """A checkerboard of supports near +1e38 and `low`, equal masses."""
    y, x = np.mgrid[0:11, 0:37]
    p = np.full((2 + bins, 11, 37), 1.0 / bins)
    up = (y + x) % 2 == 0
    p[0] = np.where(up, 0.9e38, low[0])
    p[1] = np.where(up, 1.7e38, low[1])
    return p.astype(np.float32), up


@pytest.mark.parametrize("bins", [1, 5, 8, 16])
@pytest.mark.parametrize("low", [(-1.6e38, -1.2e38), (-1.6e38, -1.6e38)])
def test_disjoint_far_supports(ucp, bins, low):
    p, up = _params(bins, low)
    dev = torch.from_numpy(p).cuda()
    ctx = ucp.Context(0)
    desc = ucp.make_desc("histogram", bins=bins)
    for types in (3, ucp.UCP_MIN, ucp.UCP_MAX):
        pmin, pmax, _ = ctx.probability_from_params(dev, desc, types)
        # masses of 1 / bins: their FP32 sum is 1 to a few units in the last place
        if types & 1:
            assert np.abs(pmin.cpu().numpy() - np.where(up, 0.0, 1.0)).max() <= 1e-5
        if types & 2:
            assert np.abs(pmax.cpu().numpy() - np.where(up, 1.0, 0.0)).max() <= 1e-5
    w = torch.ones(11, 37, device="cuda")
    for t in (ucp.UCP_MIN, ucp.UCP_MAX):
        g = ctx.backward(dev, desc, t, w)
        assert torch.isfinite(g).all()


@pytest.mark.parametrize("bins", [5, 16])
def test_support_reaching_in_from_far_below(ucp, orc, bins):
    p, _ = _params(bins, (-1.6e38, 1.2e38))
    dev = torch.from_numpy(p).cuda()
    ctx = ucp.Context(0)
    desc = ucp.make_desc("histogram", bins=bins)
    pmin, pmax, _ = ctx.probability_from_params(dev, desc)
    one = [ctx.probability_from_params(dev, desc, t)[i] for i, t in ((0, ucp.UCP_MIN),
                                                                     (1, ucp.UCP_MAX))]
    torch.cuda.synchronize()
    assert torch.equal(one[0].nan_to_num(2.0), pmin.nan_to_num(2.0))
    assert torch.equal(one[1].nan_to_num(2.0), pmax.nan_to_num(2.0))
    _, up = _params(bins, (0, 1))
    rmin, rmax, _ = orc.prob(p.astype(np.float64), 2, bins=bins)
    # (the wide supports themselves are too wide a centre: NaN)
    assert np.isnan(pmin.cpu().numpy()[~up]).all()
    assert np.abs(pmin.cpu().numpy() - rmin)[up].max() <= 1e-5
    assert np.abs(pmax.cpu().numpy() - rmax)[up].max() <= 1e-5
