"""The histogram adjoint's in-bin integrals beside a large running sum: a
neighbour's partial of a bin is C (the integral up to the bin) plus the bin's
own integral.  Here C is the centre's first bin (1.0625), and the bin's integral
comes in some sixty pieces of less than half a unit in the last place of C
each (2.4e-6 in all): added to C one by one every one of them would be lost."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
B = 16


@pytest.fixture(scope="module")
def ucp():
    from paper_2407_18015_gb300 import build
    build.build()
    from paper_2407_18015_gb300 import ucp as u
    return u


def _params(mirrored):
    p = np.zeros((2 + B, 3, 3))
    p[1], p[2:] = 1.0, 1.0 / B
    # the centre: all but 2.4e-6 of its mass (1.0625) in the first bin of [0, 1]
    p[2:, 1, 1] = 1.6e-7
    p[2, 1, 1] = 1.0625
    # three neighbours that start after that bin, nearly all mass at their end,
    # their edges and the centre's 1/64 apart
    for k, (y, x) in enumerate(((0, 1), (1, 0), (2, 1))):
        p[0, y, x], p[1, y, x] = 1 / 16 + (k + 1) / 64, 17 / 16 + (k + 1) / 64
        p[2:, y, x] = 1e-3
        p[1 + B, y, x] = 1 - 15e-3
    # the fourth: an edge at 1/16, its next beyond the centre's support
    h = 1.25
    p[0, 1, 2], p[1, 1, 2] = 1 / 16 - h, 1 / 16 + 15 * h
    if mirrored:
        p = np.concatenate([-p[1:2], -p[0:1], p[:1:-1]])
    return p.astype(np.float32)


@pytest.mark.parametrize("cptype", [1, 2])
def test_small_pieces_beside_a_large_sum(ucp, orc, cptype):
    p = _params(cptype == 2)
    w = np.zeros((3, 3), np.float32)
    w[1, 1] = 1.0
    ctx = ucp.Context(0)
    g = ctx.backward(torch.from_numpy(p).cuda(), ucp.make_desc("histogram", bins=B), cptype,
                     torch.from_numpy(w).cuda()).cpu().numpy()
    r = orc.grad(p.astype(np.float64), 2, w.astype(np.float64), cptype=cptype, bins=B)
    got, ref = ((a if cptype == 1 else a[::-1])[:, 1, 2] for a in (g, r))
    # C alone is 1.0625 (its mass), the bin's integral above 1.5e-6
    assert 1.5e-6 < ref[1] - 1.0625 < 2.4e-6
    # C: one piece of four roundings and a reciprocal of 2 units, the sum's
    # rounding: 6 units of 2^-23
    assert abs(got[1] - ref[1]) <= 6 * 2.0 ** -23
