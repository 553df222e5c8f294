"""The read-back's integer velocity quotient on the host (no GPU), at momenta on and next to powers of two.

lbm_fx_velocity_host runs the read-back kernels' route: exact integer sums S and J, rho = rho_s + S rounded to
double, and J / rho as an integer product.  Nodes here hold PDFs that the sums take exactly, so rho is within 2^-53 of
the exact density and a velocity within 2^-53 (rho) + (1/2 + 2^-4) 2^-52 (the quotient) of the exact one, relatively.
"""
from fractions import Fraction

import numpy as np
import pytest

import paper_1410_0412_gb300 as lbm
from oracle.d3q19 import C, W


def _check(d, p):
    out, ok = lbm.lbm_fx_velocity_host(d, p)
    assert ok.all()
    for n in range(len(d)):
        f = [Fraction(float(v)) for v in d[n]]
        rho = sum(f) + (Fraction(p.rho0) if p.shifted else 0)
        assert abs(Fraction(float(out[n, 0])) - rho) <= rho / 2 ** 53
        for a in range(3):
            ex = sum(int(C[i][a]) * f[i] for i in range(19)) / rho
            err = abs(Fraction(float(out[n, 1 + a])) - ex)
            assert err <= abs(ex) * Fraction(17, 16) / 2 ** 52, (n, a, float(out[n, 1 + a]), float(ex))


@pytest.mark.parametrize("pair", range(1, 10))
def test_quotient_next_to_powers_of_two_in_full_storage(pair):
    # J = +-(2^-k - m 2^-56) and +-(2^-k + m 2^-56), every term a multiple of 2^-57 of the largest PDF
    rows = []
    for k in range(4, 40):
        for m in (0, 1, 2, 5, 1 << 12, 1 << 23):
            for sign in (1, -1):
                j = 2.0 ** -k + sign * m * 2.0 ** -56
                if j <= 0:
                    continue
                for a, b in ((2 * pair - 1, 2 * pair), (2 * pair, 2 * pair - 1)):
                    d = np.full(19, 1.0 / 64)
                    d[0], d[a], d[b] = 0.75, 0.0625 + j, 0.0625
                    rows.append(d)
    _check(np.array(rows), lbm.Params(shifted=False))


@pytest.mark.parametrize("axis", range(3))
def test_quotient_next_to_powers_of_two_in_deviation_storage(axis):
    rows = []
    for k in range(3, 200, 7):
        for j in (2.0 ** -k, np.nextafter(2.0 ** -k, 0), np.nextafter(2.0 ** -k, 1)):
            for v in (j, -j):
                d = np.zeros(19)
                d[2 * axis + 1], d[0] = v, -v
                rows.append(d)
    _check(np.array(rows), lbm.Params(shifted=True))


def test_velocity_of_uniform_equilibria_at_powers_of_two():
    # momentum rho u of nominally 2^-k often lands a few ulps below it
    rows = []
    w, c = np.asarray(W, dtype=np.float64), np.asarray(C, dtype=np.float64)
    for rho in (1.0, 1.01, 0.93):
        for k in range(3, 10):
            for a in range(3):
                for v in (2.0 ** -k, -2.0 ** -k, 2.0 ** -k / rho, -2.0 ** -k / rho):
                    u = np.zeros(3)
                    u[a] = v
                    cu = c @ u
                    rows.append(w * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * (u @ u)))
    d = np.array(rows)
    out, ok = lbm.lbm_fx_velocity_host(d, lbm.Params(shifted=False))
    assert ok.all()
    for n in range(len(d)):
        f = [Fraction(float(x)) for x in d[n]]
        rho = sum(f)
        cut = 19 * max(f) / 2 ** 57  # PDFs more than 5 binades below the largest are truncated
        for a in range(3):
            ex = sum(int(C[i][a]) * f[i] for i in range(19)) / rho
            tol = abs(ex) * Fraction(17, 16) / 2 ** 52 + 2 * cut / rho
            assert abs(Fraction(float(out[n, 1 + a])) - ex) <= tol, (n, a, float(out[n, 1 + a]), float(ex))


def test_velocity_refuses_what_it_cannot_hold():
    d = np.tile(np.asarray(W, dtype=np.float64), (5, 1))
    d[0, 3], d[1, 4], d[2], d[3] = np.nan, np.inf, -d[2], 0.0  # not a number, infinite, negative density, none
    assert lbm.lbm_fx_velocity_host(d, lbm.Params(shifted=False))[1].tolist() == [False, False, False, False, True]
