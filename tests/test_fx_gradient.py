"""dJ/ds of the FP64 adjoint step's fixed-point route, on the host (no GPU), against exact rationals.

One node's term is rho times a sum of products of u with M1 = sum w c mu, with K u and with K g, K = 9 M2 - 3 M0 of the
adjoint vector mu; each may be far smaller than max|mu|: a smooth adjoint field (M1 and K small), a slow flow, a large
rest value.  Bound: u is within 2^-50 of |u| (its own products 2^-57, forward PDFs over many binades the rest), M1 and
K are exact for mu within 5 binades of its largest (19 truncations of 2^-57 max|mu| otherwise), the sums' products are
within 2^-54 and their conversions within 2^-53: 2^-50 of 4 (3 |M1| |u| + |K| |u| (|u| + |g|)), with sums of magnitudes
for |M1| and |K| and the rates' and the drag's factors below 4.
"""
from fractions import Fraction

import numpy as np
import pytest

import paper_1410_0412_gb300 as lbm
from oracle.d3q19 import C
from test_fx_adjoint import WF, _exact, _forward


def _fields(n, seed):
    rng = np.random.default_rng(seed)
    x = rng.random((n, 1))
    yield 1e-7 * rng.standard_normal((n, 19))
    yield 1e-7 * (1 + x + 1e-3 * rng.standard_normal((n, 19)))  # smooth
    yield 1e-7 * (1 + x + 1e-8 * rng.standard_normal((n, 19)))
    yield 1e-7 * (1 + x + 0 * rng.random((n, 19)))  # constant: M1 = K = 0
    yield 1e-7 * (np.asarray(C)[:, 0] + 1e-4 * rng.standard_normal((n, 19)))  # near the objective's own
    rest = 1e-9 * rng.standard_normal((n, 19))
    rest[:, 0] = 1e-3
    yield rest


def _scale(mu, u, g):
    m = [Fraction(float(v)) for v in mu]
    c = [[int(v) for v in row] for row in C]
    M0 = sum(w * v for w, v in zip(WF, m))
    M1 = [sum(WF[i] * c[i][a] * m[i] for i in range(19)) for a in range(3)]
    K = [[9 * sum(WF[i] * c[i][a] * c[i][b] * m[i] for i in range(19)) - (3 * M0 if a == b else 0) for b in range(3)]
         for a in range(3)]
    big = max(abs(v) for v in m)
    cut = 0 if all(v == 0 or abs(v) * 16 >= big for v in m) else 19 * big / 2 ** 57  # of M1; 9 times it of K
    gm = max(abs(Fraction(v)) for v in g)
    k = sum(abs(v) for row in K for v in row)
    full = 4 * (3 * sum(abs(v) for v in M1) * u + k * u * (u + gm))
    return full / 2 ** 50 + 4 * cut * u * (3 + 9 * 9 * (u + gm))


@pytest.mark.parametrize("shifted", [False, True])
@pytest.mark.parametrize("omega,g", [(1.0, (1e-6, 0.0, 0.0)), (1.0, (0.0, 0.0, 0.0)), (0.8, (1e-7, -3e-8, 2e-9)),
                                     (1.9, (1e-4, 0.0, 0.0))])
@pytest.mark.parametrize("drag", [False, True])
def test_gradient_keeps_its_own_accuracy(shifted, omega, g, drag):
    n = 8
    p = lbm.Params(omega_plus=omega, magic=3 / 16, g=g, shifted=shifted)
    s = np.linspace(0.0, 1.0, n, dtype=np.float32) if drag else None
    for umax in (1e-2, 1e-4, 1e-6):
        d = _forward(n, 4, shifted, umax)
        if not shifted:  # u itself is within 2^-50 of the PDFs' size there, not of |u|
            d = d if umax == 1e-2 else _forward(n, 4, shifted, 1e-2)
        for mu in _fields(n, 3):
            _, grad, ok = lbm.lbm_fx_adjoint_host(d, mu, p, s)
            assert ok.all()
            for k in range(n):
                _, ex, rho, u = _exact(d[k], mu[k], p, 0.0 if s is None else s[k])
                assert abs(Fraction(float(grad[k])) - ex) <= rho * _scale(mu[k], u, g) + abs(ex) / 2 ** 51, (umax, k)


def test_constant_field_has_no_gradient():
    # M1 and K vanish exactly, so the term has to
    p = lbm.Params(omega_plus=1.0, magic=3 / 16, g=(1e-6, 0.0, 0.0), shifted=True)
    mu = np.full((6, 19), 1.0) * np.array([[1.0], [-3.5], [1e-9], [7e5], [1 / 3], [0.0]])
    _, grad, ok = lbm.lbm_fx_adjoint_host(_forward(6, 4, True, 0.01), mu, p, np.full(6, 0.5, np.float32))
    assert ok.all() and (grad == 0).all()


@pytest.mark.parametrize("u", [1e-30, 1e-90, 1e-140, 1e-200, 1e-280])
def test_the_slowest_flows_stay_in_the_range(u):
    # a front that runs into a fluid at rest: terms quadratic in u underflow, the linear one still counts
    p = lbm.Params(omega_plus=1.0, magic=3 / 16, g=(0.0, 0.0, 0.0), shifted=True)
    d = np.zeros((3, 19))
    d[:, 1], d[:, 4], d[:, 7] = u, -0.7 * u, 0.2 * u
    mu = np.random.default_rng(3).standard_normal((3, 19))
    _, grad, ok = lbm.lbm_fx_adjoint_host(d, mu, p, np.full(3, 0.5, np.float32))
    assert ok.all()
    for k in range(3):
        _, ex, rho, um = _exact(d[k], mu[k], p, 0.5)
        assert abs(Fraction(float(grad[k])) - ex) <= rho * _scale(mu[k], um, p.g) + abs(ex) / 2 ** 51
