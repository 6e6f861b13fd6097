"""The histogram row walks from parameters: one type alone, both types and the
oracle, with point-mass neighbours (whose survival jumps inside the walk),
masses that do not sum to 1, lines and ragged tiles, at the row bounds' edges
(8 | 9 and 16 bins)."""
import numpy as np
import pytest
import torch

import helpers as H_

pytestmark = pytest.mark.gpu
TOL = 1e-5


@pytest.fixture(scope="module")
def ucp():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2407_18015_gb300 import build
    build.build()
    from paper_2407_18015_gb300 import ucp as u
    return u


def _params(Hh, Ww, bins, seed, scale):
    rng = np.random.default_rng(seed)
    p = H_.random_params(2, Hh, Ww, rng, bins=bins)
    p[2:] *= rng.uniform(0.5, 1.5, (Hh, Ww))
    pm = rng.random((Hh, Ww)) < 0.15
    p[1][pm] = p[0][pm]
    tie = rng.random((Hh, Ww)) < 0.1               # equal supports: every edge ties
    p[0][tie], p[1][tie] = -0.5, 0.75
    p[:2] *= scale
    return p.astype(np.float32)


@pytest.mark.parametrize("bins", [1, 2, 5, 8, 9, 16])
@pytest.mark.parametrize("shape,boundary,scale", [((9, 33), 0, 1.0), ((17, 65), 1, 1e-12),
                                                  ((1, 70), 0, 1e9), ((40, 31), 0, 1.0)])
def test_one_type_equals_both_and_oracle(ucp, orc, bins, shape, boundary, scale):
    p = _params(*shape, bins, seed=bins * 100 + shape[1], scale=scale)
    dev = torch.from_numpy(p).cuda()
    ctx = ucp.Context(0)
    desc = ucp.make_desc("histogram", bins=bins, boundary=boundary)
    pmin, pmax, st = ctx.probability_from_params(dev, desc)
    only_min, _, st1 = ctx.probability_from_params(dev, desc, ucp.UCP_MIN)
    _, only_max, st2 = ctx.probability_from_params(dev, desc, ucp.UCP_MAX)
    torch.cuda.synchronize()
    assert torch.equal(only_min, pmin) and torch.equal(only_max, pmax)
    assert torch.equal(st1, st) and torch.equal(st2, st)
    rmin, rmax, rst = orc.prob(p.astype(np.float64), 2, bins=bins, boundary=boundary)
    # masses sum to at most 1.5: tolerances scale with the product of five totals
    assert np.abs(pmin.cpu().numpy() - rmin).max() <= TOL * 1.5 ** 5
    assert np.abs(pmax.cpu().numpy() - rmax).max() <= TOL * 1.5 ** 5
    np.testing.assert_array_equal(st.cpu().numpy(), rst)
    sad, _ = ctx.saddle_from_params(dev, desc)
    rsad = orc.saddle(p.astype(np.float64), 2, bins=bins)[0]
    assert np.abs(sad.cpu().numpy() - rsad).max() <= 2 * TOL * 1.5 ** 5
