"""The larger stencils' histogram pieces (CPU, rational arithmetic): the mean of
a product of six or eight linear factors from pairs of factors is the integral
over the piece."""
import random
from fractions import Fraction as Fr
from math import comb

import pytest


def _pairs(L, R):
    """The mean over [0, 1] of prod (L_i + (R_i - L_i) t)."""
    K = len(L)
    b = [(L[j] * L[j + 1], L[j] * R[j + 1] + R[j] * L[j + 1], R[j] * R[j + 1])
         for j in range(0, K, 2)]

    def quartic(x, y):
        return [sum(x[i] * y[k - i] for i in range(3) if 0 <= k - i < 3) for k in range(5)]

    c, d = quartic(b[0], b[1]), quartic(b[2], b[3]) if K == 8 else b[2]
    return sum(ck * dl / ((K + 1) * comb(K, k + l))
               for k, ck in enumerate(c) for l, dl in enumerate(d))


@pytest.mark.parametrize("K", [6, 8])
def test_pairs_form_is_the_integral(K):
    rng = random.Random(K)
    for _ in range(50):
        L, R = ([Fr(rng.randint(0, 64), 64) for _ in range(K)] for _ in range(2))
        poly = [Fr(1)]
        for l, r in zip(L, R):
            poly = [(poly[k] if k < len(poly) else 0) * l
                    + (poly[k - 1] if k else 0) * (r - l) for k in range(len(poly) + 1)]
        exact = sum(c / (k + 1) for k, c in enumerate(poly))
        assert _pairs(L, R) == exact
