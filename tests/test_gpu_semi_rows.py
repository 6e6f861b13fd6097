"""The semianalytical estimator's row layout and bin search at bins that are
and are not powers of two (1 to 64), odd sample counts, point-mass
neighbours, empty bins and lines, against the oracle on identical streams."""
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


@pytest.mark.parametrize("B", [1, 2, 3, 5, 8, 15, 16, 17, 64])
@pytest.mark.parametrize("shape,S", [((10, 35), 33), ((1, 40), 2), ((9, 33), 1)])
def test_semi_rows(ucp, orc, B, shape, S):
    rng = np.random.default_rng(B * 7 + S)
    p = H_.random_params(2, *shape, rng, bins=B)
    p[2:][rng.random(p[2:].shape) < 0.3] = 0.0     # empty bins
    pm = rng.random(shape) < 0.2
    p[1][pm] = p[0][pm]
    p32 = p.astype(np.float32)
    ctx = ucp.Context(0)
    desc = ucp.make_desc("histogram_semi", bins=B, mc_samples=S, seed=77, field_id=1)
    dev = torch.from_numpy(p32).cuda()
    pmin, pmax, _ = ctx.probability_from_params(dev, desc)
    sad, _ = ctx.saddle_from_params(dev, desc)
    torch.cuda.synchronize()
    idx = np.arange(shape[0] * shape[1])
    ref = orc.semi_at(p32.astype(np.float64), B, idx, S, 77, field=1)
    for g, r in zip((pmin, pmax, sad), ref):
        assert np.abs(g.cpu().numpy().ravel() - r).max() <= 1e-5
