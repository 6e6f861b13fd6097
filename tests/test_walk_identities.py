"""Exact-arithmetic checks of the piece integrals of the histogram walks (CPU,
rational arithmetic): products of linear factors f_i = l_i + D_i t.

- forward walk: int_0^1 f_0 f_1 f_2 f_3 = (f(0) + 4 f(1/2) + f(1)) / 6
  - D_0 D_1 D_2 D_3 / 120;
- adjoint walk: with f_i = m_i - E_i s, s in [-1, 1], p = m_0 m_1, e = E_0
  E_1, b = m_0 E_1 + m_1 E_0, q, g, c likewise for factors 2 and 3, U = q +
  g/3, V = q/3 + g/5: the mean of the product is p U + e V + b c / 3, the mean
  of f_1 f_2 f_3 is m_1 U + E_1 c / 3, and its mean against a linear weight
  w - v s adds v (m_1 c / 3 + E_1 V).
"""
import random
from fractions import Fraction as Fr


def _poly(factors):
    out = [Fr(1)]
    for c0, c1 in factors:
        nxt = [Fr(0)] * (len(out) + 1)
        for k, c in enumerate(out):
            nxt[k] += c * c0
            nxt[k + 1] += c * c1
        out = nxt
    return out


def _integral(factors, a, b):
    return sum(c * (Fr(b) ** (k + 1) - Fr(a) ** (k + 1)) / (k + 1)
               for k, c in enumerate(_poly(factors)))


def _values(rng, n):
    return [Fr(rng.randint(0, 64), 64) for _ in range(n)]


def test_simpson_with_fourth_order_term():
    rng = random.Random(11)
    for _ in range(200):
        l, r = _values(rng, 4), _values(rng, 4)
        D = [b - a for a, b in zip(l, r)]
        f0 = f1 = fm = dd = Fr(1)
        for a, b, d in zip(l, r, D):
            f0, f1, fm, dd = f0 * a, f1 * b, fm * (a + b) / 2, dd * d
        assert (f0 + 4 * fm + f1) / 6 - dd / 120 == _integral(list(zip(l, D)), 0, 1)


def test_middle_value_forms():
    rng = random.Random(12)
    for _ in range(200):
        m, E = _values(rng, 4), _values(rng, 4)
        w, v = _values(rng, 2)
        f = [(a, -d) for a, d in zip(m, E)]
        p, e, b = m[0] * m[1], E[0] * E[1], m[0] * E[1] + m[1] * E[0]
        q, g, c = m[2] * m[3], E[2] * E[3], m[2] * E[3] + m[3] * E[2]
        U, V = q + g / 3, q / 3 + g / 5
        assert p * U + e * V + b * c / 3 == _integral(f, -1, 1) / 2
        loo = m[1] * U + E[1] * c / 3
        assert loo == _integral(f[1:], -1, 1) / 2
        weighted = w * loo + v * (m[1] * c / 3 + E[1] * V)
        assert weighted == _integral(f[1:] + [(w, -v)], -1, 1) / 2
