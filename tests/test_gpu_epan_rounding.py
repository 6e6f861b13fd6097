"""The Epanechnikov pieces' rounding: the mean error against 64 bits is that of
the arithmetic they document, restated here in numpy binary32 (each node forms
every factor's argument anew; the piece's middle and the reciprocal of the
centre's width in two floats).  Arguments whose rounding is common to all nodes
of a piece have a mean error 15 % larger.  8 % cover the kernel's approximate
reciprocals (2 units in the last place) and the order of its sums."""
import numpy as np
import pytest
import torch
from numpy.polynomial.legendre import leggauss

pytestmark = pytest.mark.gpu
f32 = np.float32


@pytest.fixture(scope="module")
def ucp():
    from paper_2407_18015_gb300 import build
    build.build()
    from paper_2407_18015_gb300 import ucp as u
    return u


def _fma(a, b, c):
    return (np.asarray(a, np.float64) * b + c).astype(f32)


def _minimum32(m, w):
    """P_min in binary32 of centres m[0], w[0] with neighbours m[1:], w[1:]."""
    w1, dn, iw = w[0], m[1:] - m[0], f32(1) / w[1:]
    R, L = np.minimum(w1, (dn + w[1:]).min(0)), -w1
    t = np.clip(dn - w[1:], L, R)
    o = np.argsort(t, 0, kind="stable")
    d, iw = np.take_along_axis(dn, o, 0), np.take_along_axis(iw, o, 0)
    x = np.concatenate([L[None], np.take_along_axis(t, o, 0), R[None]])
    hi = f32(1) / w1
    lo = hi * _fma(-w1, hi, f32(1))
    acc, comp = np.zeros_like(w1), np.zeros_like(w1)
    for J, n in enumerate((2, 3, 5, 6, 8)):
        half, mid = f32(0.5) * (x[J + 1] - x[J]), f32(0.5) * (x[J] + x[J + 1])
        merr = (x[J] - mid) + half
        s = [np.zeros_like(w1), np.zeros_like(w1)]     # nodes in pairs, an odd last one on top
        for k, (xi, wt) in enumerate(zip(*(a.astype(f32) for a in leggauss(n)))):
            xx = _fma(half, xi, merr) + mid
            u = _fma(xx, hi, xx * lo)
            Q, T = np.ones_like(w1), np.ones_like(w1)
            for i in range(J):
                q = _fma(d[i] - xx, iw[i], f32(1))
                Q, T = Q * q, T * (f32(3) - q)
            f = (Q * Q) * (T * _fma(-u, u, f32(1)))
            if k + 1 == n and n % 2:
                s = [_fma(wt, f, s[0] + s[1]), f32(0)]
            else:
                s[k % 2] = _fma(wt, f, s[k % 2])
        y = np.where(half > 0, (s[0] + s[1]) * (half * f32(0.25 ** J)), f32(0)) - comp
        tot = acc + y
        comp, acc = (tot - acc) - y, tot
    r = f32(0.75) * acc
    return np.where(R > L, np.maximum(_fma(r, hi, r * lo), 0), 0)


def test_mean_error_of_the_documented_arithmetic(ucp, orc):
    H, W = 202, 202
    rng = np.random.default_rng(3)
    p = np.stack([rng.normal(0, 0.1, (H, W)), rng.uniform(0.8, 1.2, (H, W))]).astype(f32)
    m, w = (np.stack([a[1:-1, 1:-1], a[1:-1, 2:], a[:-2, 1:-1], a[1:-1, :-2], a[2:, 1:-1]])
            for a in p)
    shape = m.shape[1:]
    m, w = m.reshape(5, -1), w.reshape(5, -1)
    rmin, rmax, _ = orc.prob(p.astype(np.float64), 1)
    ctx = ucp.Context(0)
    pmin, pmax, _ = ctx.probability_from_params(torch.from_numpy(p).cuda(),
                                                ucp.make_desc("epanechnikov"))
    with np.errstate(all="ignore"):
        want = [_minimum32(s * m, w).reshape(shape) for s in (f32(1), f32(-1))]
    for g, e, r in zip((pmin, pmax), want, (rmin, rmax)):
        err = np.abs(g.cpu().numpy() - r)[1:-1, 1:-1].mean()
        assert err <= 1.08 * np.abs(e - r[1:-1, 1:-1]).mean()
