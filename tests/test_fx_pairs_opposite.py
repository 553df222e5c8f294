"""The fixed-point pair update at pairs of opposite signs next to the scale's limit, on the host (no GPU).

|d_a - d_b| reaches 4 B for PDFs of opposite signs next to 2 B; 2^4 times that is 2^63 units, past what a factor of the
update's product holds.  Every value stays within 8 units of the pair scale, which is reported, plus half an ulp.
"""
from fractions import Fraction

import numpy as np
import pytest

import paper_1410_0412_gb300 as lbm
from test_fx_pairs import _exact_pairs


@pytest.mark.parametrize("lp1", [True, False])
def test_opposite_pairs_up_to_the_largest_difference(lp1):
    rows = []
    for k in range(1, 10):
        for gap in (0.5, 2.0 ** -10, 2.0 ** -26, 2.0 ** -28, 2.0 ** -40, 2.0 ** -53):
            for sign in (1.0, -1.0):
                d = np.full(19, 1.0 / 36)
                d[2 * k - 1], d[2 * k] = sign * (1 - gap), -sign * (1 - gap)
                rows.append(d)
    d = np.array(rows)
    terms = np.random.default_rng(2).uniform(-0.1, 0.1, (len(d), 10))
    out, ok = lbm.lbm_fx_pairs_host(d, terms, -1.0 / 14.0, 0.0 if lp1 else 0.125, lp1)
    assert ok.all()
    for n in range(len(d)):
        ex = _exact_pairs(d[n], terms[n], -1.0 / 14.0, 0.0 if lp1 else 0.125)
        unit = Fraction(2) ** (int(out[n, 0]) - 1080)
        for i in range(1, 19):
            err = abs(Fraction(float(out[n, i])) - ex[i])
            assert err <= 8 * unit + Fraction(float(np.spacing(abs(out[n, i])))) / 2, (n, i, float(err))


@pytest.mark.parametrize("omega", [1.0, 0.8])
def test_collision_of_opposite_pairs_is_right_or_refused(omega):
    import test_fx_collide
    rows = []
    for k in range(1, 10):
        for gap in (0.5, 2.0 ** -20, 2.0 ** -26, 2.0 ** -30, 2.0 ** -53):
            d = np.full(19, 1.0 / 36)  # the other pairs cancel most of this one's momentum
            d[0], d[2 * k - 1], d[2 * k] = 0.9, 1 - gap, -(1 - gap)
            for m in range(1, 10):
                if m != k:
                    d[2 * m - 1], d[2 * m] = 0.02, 0.03
            rows.append(d)
    test_fx_collide._check(np.array(rows), lbm.Params(omega_plus=omega, g=(0.0, 0.0, 0.0), shifted=False), None)
