"""The FP64 step's whole collision in fixed point, run on the host (no GPU).

The LBM_F64 step kernels evaluate the TRT collision with Guo forcing (Sect. 2)
from exact integer moments: the momentum q = rho u, the force F = rho g - s q,
the class terms K0, T and O and the nine pairs are 64-bit fixed-point values at
a scale 2^(es - 1080), es = emax - kx, tied to the node's largest PDF (emax its
biased exponent).  lbm_fx_collide_host runs the same routines on the host.

Bound, from the routines' steps in units of that scale (each product is within
3/4 of a unit, each truncation within 1): q 6, F 10 (both with drag), T 10,
O 6, u 8 Q64 units, K0 3; (c.u)(c.T) then 14, and p = K0 + (c.u)(c.T) + c.O +
the exact pair parts at most 40, plus one rounding to double.  PDFs more than
5 binades below the largest are truncated at 2^kx units each: at most 16 2^kx
more.  Deviation storage rounds rho to double: 2^-52 of (c.u)(c.T) more.
"""
import itertools
from fractions import Fraction

import numpy as np
import pytest

import paper_1410_0412_gb300 as lbm
from oracle.d3q19 import C, W

RHO0 = 1.0


def _biased(x):
    return int(np.frexp(abs(x))[1]) - 1 + 1023 if x != 0 else 0


def _exact(d, p, s):
    """Post-collision PDFs in exact rationals, and the largest |(c.u)(c.T)|; the collision's constants (l+/18,
    l-/6, a-/6, the rates and 1 - l+-, halved) are the doubles that the library forms."""
    rho_s = Fraction(p.rho0) if p.shifted else Fraction(0)
    f = [Fraction(float(v)) for v in d]
    lp = p.omega_plus
    lm = 1.0 / (p.magic / (1.0 / lp - 0.5) + 0.5)
    k0a, k1, k2 = Fraction(lp / 18.0), Fraction(lp) / 4, Fraction(lm / 6.0)
    fs, fo = Fraction(1.0 - lp / 2) / 2, Fraction((1.0 - lm / 2) / 6.0)
    qp, qm = Fraction((1.0 - lp) / 2), Fraction((1.0 - lm) / 2)
    g = [Fraction(v) for v in p.g]
    s = Fraction(float(np.float32(s)))
    drho = sum(f)
    rho = rho_s + drho
    J = [sum(int(C[i][a]) * f[i] for i in range(19)) for a in range(3)]
    q = [(J[a] + rho * g[a] / 2) / (1 + s / 2) for a in range(3)]
    u = [v / rho for v in q]
    F = [rho * g[a] - s * q[a] for a in range(3)]
    T = [k1 * q[a] + fs * F[a] for a in range(3)]
    O = [k2 * q[a] + fo * F[a] for a in range(3)]
    K0 = k0a * drho - sum(u[a] * T[a] for a in range(3)) / 3
    out, big = [2 * qp * f[0] + 6 * K0] + [None] * 18, Fraction(0)
    for k in range(1, 10):
        a, b = 2 * k - 1, 2 * k
        c = [int(v) for v in C[a]]
        h = Fraction(1) if k <= 3 else Fraction(1, 2)
        prod = sum(c[i] * u[i] for i in range(3)) * sum(c[i] * T[i] for i in range(3))
        even = h * (K0 + prod) + qp * (f[a] + f[b])
        odd = h * sum(c[i] * O[i] for i in range(3)) + qm * (f[a] - f[b])
        out[a], out[b] = even + odd, even - odd
        big = max(big, abs(prod))
    return out, big


def _nodes(n, seed, shifted, noise=0.05, umax=0.1):
    rng = np.random.default_rng(seed)
    w = np.asarray(W, dtype=np.float64)
    rho = 1 + 0.02 * (rng.random(n) - 0.5)
    u = 2 * umax * (rng.random((n, 3)) - 0.5)
    cu = u @ np.asarray(C, dtype=np.float64).T
    feq = w * rho[:, None] * (1 + 3 * cu + 4.5 * cu ** 2 - 1.5 * (u * u).sum(1)[:, None])
    d = feq * (1 + noise * (rng.random((n, 19)) - 0.5))
    return d - w * RHO0 if shifted else d


def _check(d, p, s):
    out, ok = lbm.lbm_fx_collide_host(d, p, s)
    for n in np.nonzero(ok)[0]:
        ex, big = _exact(d[n], p, 0.0 if s is None else s[n])
        e = [_biased(v) for v in d[n]]
        emin = max([64] + ([_biased(p.rho0 * v) for v in p.g] if p.shifted else []))
        emax = max(e + [emin])
        near = (d[n] > 0).all() and max(e) - min(e) <= 5 and min(e) >= 64
        kx = 0 if p.shifted else 4 if near and p.omega_plus == 1.0 else 2
        unit = Fraction(2) ** (emax - kx - 1080)
        tol = 40 * unit + (0 if emax - min(e) <= 5 else 16 * 2 ** kx * unit)
        if p.shifted:
            tol += big / 2 ** 52
        for i in range(19):
            err = abs(Fraction(float(out[n, i])) - ex[i])
            assert err <= tol + Fraction(float(np.spacing(abs(out[n, i])))) / 2, (n, i, float(err / unit))
    return ok


@pytest.mark.parametrize("shifted,omega,g,drag", list(itertools.product(
    [False, True], [1.0, 0.8, 1.9], [(0.0, 0.0, 0.0), (1e-6, 0.0, 0.0), (1e-4, -3e-5, 2e-5)], [False, True])))
def test_fx_collide_within_bound_of_exact_rationals(shifted, omega, g, drag):
    p = lbm.Params(omega_plus=omega, magic=3 / 16, g=g, rho0=RHO0, shifted=shifted)
    d = _nodes(40, 5, shifted)
    s = np.linspace(0.0, 1.0, 40, dtype=np.float32) if drag else None
    assert _check(d, p, s).all()


@pytest.mark.parametrize("shifted", [False, True])
@pytest.mark.parametrize("omega", [1.0, 1.6])
def test_fx_collide_edges_of_its_range(shifted, omega):
    # where it accepts a node the result is right, however odd the node: PDFs over many binades and signs,
    # velocities around the 1/4 limit, densities next to a power of two, forces from tiny to out of range
    rng = np.random.default_rng(17)
    n, accepted, refused = 60, 0, 0
    s = rng.random(n).astype(np.float32)
    for g in ((0.0, 0.0, 0.0), (1e-30, 0.0, 0.0), (3e-3, 2e-9, -1e-3), (0.7, 0.0, 0.0), (-40.0, 2.0, 1e6)):
        p = lbm.Params(omega_plus=omega, magic=3 / 16, g=g, rho0=RHO0, shifted=shifted)
        for d in (_nodes(n, 1, shifted, umax=0.26), _nodes(n, 2, shifted, noise=1.9, umax=0.01),
                  _nodes(n, 3, shifted, noise=1e-12, umax=1e-13) * (1 + 1e-14 * rng.standard_normal((n, 1))),
                  _nodes(n, 4, shifted) * 2.0 ** rng.integers(-40, 40, (n, 1)),
                  rng.standard_normal((n, 19)) * 2.0 ** rng.integers(-30, 2, (n, 19))):
            for q in (None, s):
                ok = _check(d, p, q)
                accepted, refused = accepted + ok.sum(), refused + (~ok).sum()
    assert accepted > 500 and refused > 100


def test_fx_collide_refuses_what_it_cannot_hold():
    d = _nodes(6, 9, False)
    p = lbm.Params(omega_plus=1.0, g=(1e-6, 0.0, 0.0), shifted=False)
    s = np.array([0.5, 1.5, -0.1, np.nan, 1.0, 0.0], np.float32)
    assert lbm.lbm_fx_collide_host(d, p, s)[1].tolist() == [True, False, False, False, True, True]
    bad = d.copy()
    bad[0, 4], bad[1, 0], bad[2] = np.nan, np.inf, -bad[2]  # not a number, infinite, negative density
    ok = lbm.lbm_fx_collide_host(bad, p)[1]
    assert not ok[:3].any() and ok[3:].all()
