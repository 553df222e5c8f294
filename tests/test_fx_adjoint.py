"""The FP64 adjoint step's arithmetic in fixed point, run on the host (no GPU), against exact rationals.

lambda_n = (dC/dF)^T mu and dJ/ds of one node, with C the TRT collision: the exact values follow from the weighted
moments of mu (M0, M1, M2) as the adjoint kernel's header states them.  In units 2^(em - 1080) of mu's scale (em the
largest biased exponent of mu) the routine's products give at most 40, and its constants, doubles like those of the
FP64 form, 2^-53 of terms up to 2^59 units each: 128 units in all, plus the rounding of the result.  dJ/ds is carried
p bits finer, 2^-p <= 64 |u|: 40 units there, rho |u| max|mu| 2^-45 in all.  Forward PDFs more than 5 binades below
the largest lose 2^-57 of it each, which moves u, and so each result, by less than 2^-50 of its scale.
"""
import itertools
from fractions import Fraction

import numpy as np
import pytest

import paper_1410_0412_gb300 as lbm
from oracle.d3q19 import C, W

WF = [Fraction(1, 3)] + [Fraction(1, 18)] * 6 + [Fraction(1, 36)] * 12


def _exact(d, mu, p, s):
    lp = Fraction(p.omega_plus)
    lm = Fraction(1.0 / (p.magic / (1.0 / p.omega_plus - 0.5) + 0.5))
    ap, am = 1 - lp / 2, 1 - lm / 2
    f, m = [Fraction(float(v)) for v in d], [Fraction(float(v)) for v in mu]
    g, s = [Fraction(v) for v in p.g], Fraction(float(np.float32(s)))
    rho = sum(f) + (Fraction(p.rho0) if p.shifted else 0)
    kd = 1 / (1 + s / 2)
    c = [[int(v) for v in row] for row in C]
    u = [kd * (sum(c[i][a] * f[i] for i in range(19)) / rho + g[a] / 2) for a in range(3)]
    M0 = sum(w * v for w, v in zip(WF, m))
    M1 = [sum(WF[i] * c[i][a] * m[i] for i in range(19)) for a in range(3)]
    M2 = [[sum(WF[i] * c[i][a] * c[i][b] * m[i] for i in range(19)) for b in range(3)] for a in range(3)]
    dot = lambda x, y: sum(x[a] * y[a] for a in range(3))
    M2u, M2g = [dot(M2[a], u) for a in range(3)], [dot(M2[a], g) for a in range(3)]
    uu, q, av = dot(u, u), dot(u, M2u), dot(M1, u)
    ds = -9 * ap * q + 3 * ap * M0 * uu - 3 * am * av
    psi = (lp * M0 * (1 - uu * 3 / 2) + lp * q * 9 / 2 + 3 * lm * av + 9 * ap * dot(u, M2g) + 3 * am * dot(M1, g)
           - 3 * ap * M0 * dot(u, g) + s * ds)
    P = [-3 * lp * M0 * u[a] + 9 * lp * M2u[a] + 3 * lm * M1[a] + 9 * ap * M2g[a] - 3 * ap * M0 * g[a]
         + s * (-18 * ap * M2u[a] + 6 * ap * M0 * u[a] - 3 * am * M1[a]) for a in range(3)]
    A = psi - sum(P[a] * (u[a] - kd * g[a] / 2) for a in range(3))
    lam = [A + (1 - lp) * m[0]] + [None] * 18
    for k in range(1, 10):
        a, b = 2 * k - 1, 2 * k
        odd = (1 - lm) / 2 * (m[a] - m[b]) + kd * dot(c[a], P)
        even = A + (1 - lp) / 2 * (m[a] + m[b])
        lam[a], lam[b] = even + odd, even - odd
    return lam, rho * (ds - kd / 2 * dot(P, u)), rho, max(abs(v) for v in u)


def _forward(n, seed, shifted, umax):
    rng = np.random.default_rng(seed)
    w = np.asarray(W, dtype=np.float64)
    rho = 1 + 0.02 * (rng.random(n) - 0.5)
    u = 2 * umax * (rng.random((n, 3)) - 0.5)
    cu = u @ np.asarray(C, dtype=np.float64).T
    d = w * rho[:, None] * (1 + 3 * cu + 4.5 * cu ** 2 - 1.5 * (u * u).sum(1)[:, None])
    d = d * (1 + 0.02 * min(1.0, umax) * (rng.random((n, 19)) - 0.5))
    return d - w if shifted else d


def _check(d, mu, p, s):
    lam, grad, ok = lbm.lbm_fx_adjoint_host(d, mu, p, s)
    for n in np.nonzero(ok)[0]:
        ex, gs, rho, umax = _exact(d[n], mu[n], p, 0.0 if s is None else s[n])
        top = max(abs(float(v)) for v in mu[n])
        em = max(200, int(np.frexp(top)[1]) - 1 + 1023 if top else 0)
        tol = 128 * Fraction(2) ** (em - 1080)
        for i in range(19):
            err = abs(Fraction(float(lam[n, i])) - ex[i])
            assert err <= tol + Fraction(float(np.spacing(abs(lam[n, i])))), (n, i, float(err / tol))
        err = abs(Fraction(float(grad[n])) - gs)
        assert err <= rho * umax * Fraction(2) ** (em - 1022 - 45) + abs(gs) / 2 ** 50, (n, float(err / abs(gs)) if gs else err)
    return ok


@pytest.mark.parametrize("shifted,omega,g,drag", list(itertools.product(
    [False, True], [1.0, 0.8, 1.9], [(0.0, 0.0, 0.0), (1e-6, 0.0, 0.0), (1e-4, -3e-5, 2e-5)], [False, True])))
def test_fx_adjoint_within_bound_of_exact_rationals(shifted, omega, g, drag):
    p = lbm.Params(omega_plus=omega, magic=3 / 16, g=g, shifted=shifted)
    rng = np.random.default_rng(3)
    n = 16
    s = np.linspace(0.0, 1.0, n, dtype=np.float32) if drag else None
    for umax in (0.1, 1e-3, 1e-7):
        mu = 1e-7 * (rng.standard_normal((n, 19)) + 0.3)
        assert _check(_forward(n, 4, shifted, umax), mu, p, s).all()


@pytest.mark.parametrize("shifted", [False, True])
@pytest.mark.parametrize("omega", [1.0, 1.6])
def test_fx_adjoint_edges_of_its_range(shifted, omega):
    rng = np.random.default_rng(11)
    n, accepted, refused = 24, 0, 0
    s = rng.random(n).astype(np.float32)
    mus = (np.zeros((n, 19)), np.ones((n, 19)), -np.ones((n, 19)), rng.choice([-1.999, 1.999], (n, 19)),
           rng.standard_normal((n, 19)) * 2.0 ** rng.integers(-60, 60, (n, 19)), 1e-290 * rng.standard_normal((n, 19)))
    for g in ((0.0, 0.0, 0.0), (1e-30, 0.0, 0.0), (3e-3, 2e-9, -1e-3), (0.7, 0.0, 0.0)):
        p = lbm.Params(omega_plus=omega, magic=3 / 16, g=g, shifted=shifted)
        zero = np.zeros((n, 19)) + (0.0 if shifted else np.asarray(W))
        for d in (_forward(n, 1, shifted, 0.3), _forward(n, 2, shifted, 1e-12), zero):
            for mu in mus:
                for q in (None, s):
                    ok = _check(d, mu, p, q)
                    accepted, refused = accepted + ok.sum(), refused + (~ok).sum()
    assert accepted > 1000 and refused > 100


def test_fx_adjoint_refuses_what_it_cannot_hold():
    p = lbm.Params(g=(1e-6, 0.0, 0.0))
    d, mu = _forward(5, 9, False, 0.05), np.ones((5, 19))
    d[0, 2], d[1] = np.inf, -d[1]
    mu[2, 5] = np.nan
    assert lbm.lbm_fx_adjoint_host(d, mu, p)[2].tolist() == [False, False, False, True, True]
