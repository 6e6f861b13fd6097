"""Epanechnikov neighbours of subnormal width, whose reciprocal is beyond the
float range: they act as the point masses that they all but are.  Minimum,
maximum, saddle, larger stencils and gradient at the vertices of ordinary
width, against the oracle."""
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


def _params(width, m0):
    """Ordinary vertices with one vertex of the given width at every 4th
    column and 3rd row (so that no two of them are neighbours)."""
    H, W = 12, 37
    rng = np.random.default_rng(5)
    p = np.stack([rng.normal(0, 0.3, (H, W)), rng.uniform(0.4, 1, (H, W))]).astype(np.float32)
    tiny = np.zeros((H, W), bool)
    tiny[1::3, 2::4] = True
    p[0][tiny] = rng.uniform(-0.3, 0.3, tiny.sum()) * m0
    p[1][tiny] = np.float32(width)
    return p, tiny


@pytest.mark.parametrize("width", [1e-45, 1e-40, 2.9e-39, 1e-30])
@pytest.mark.parametrize("m0", [1.0, 0.0])
def test_subnormal_width_neighbours(ucp, orc, width, m0):
    p, tiny = _params(width, m0)
    p64 = p.astype(np.float64)
    dev = torch.from_numpy(p).cuda()
    ctx = ucp.Context(0)
    ok = ~tiny
    got = [ctx.probability_from_params(dev, ucp.make_desc("epanechnikov", stencil=s))[:2]
           for s in (0, 1, 2)]
    ref = [orc.prob(p64, 1)[:2]] + [orc.prob_stencil(p64, 1, s)[:2] for s in (1, 2)]
    got.append(ctx.saddle_from_params(dev, ucp.make_desc("epanechnikov"))[:1])
    ref.append(orc.saddle(p64, 1)[:1])
    for gs, rs in zip(got, ref):
        for g, r in zip(gs, rs):
            assert np.abs(g.cpu().numpy() - r)[ok].max() <= 1e-5


@pytest.mark.parametrize("cptype", [1, 2])
def test_gradient_beside_a_subnormal_width(ucp, orc, cptype):
    # narrow vertices on the border alone, where the interior rule takes no
    # probability: the others' gradients have no partial of a narrow centre
    p, _ = _params(1.0, 1.0)
    border = np.zeros(p.shape[1:], bool)
    border[0], border[-1] = True, True
    border[:, 0], border[:, -1] = True, True
    p[1][border] = 1e-40
    p64 = p.astype(np.float64)
    wt = np.random.default_rng(9).uniform(0, 1, p.shape[1:]).astype(np.float32)
    ctx = ucp.Context(0)
    desc = ucp.make_desc("epanechnikov", boundary=1)
    g = ctx.backward(torch.from_numpy(p).cuda(), desc, cptype,
                     torch.from_numpy(wt).cuda()).cpu().numpy()
    r = orc.grad(p64, 1, wt.astype(np.float64), cptype=cptype, boundary=1)
    ok = ~border
    assert (np.abs(g - r) <= 1e-4 * np.abs(r) + 2e-5 * max(1.0, np.abs(r[:, ok]).max()))[:, ok].all()
