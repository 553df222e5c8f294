"""Density, velocity and canonical PDFs read back from a grid, at the values where the integer routes can go wrong.

The read-back kernels form rho and u from exact integer sums of the stored PDFs and integer quotients, and widen
floats to doubles by their bits.  They are held to exact rationals on grids of any values: at rest (zero
deviations), small deviations, PDFs over many binades, subnormal ones, negative and zero densities, Inf and NaN.

Tolerance: rho is rounded twice (2^-52), a velocity component by its quotient, rho, the force and the drag factor
(2^-50 of |j / rho| + |g / 2|); FP64 PDFs more than 5 binades below the largest lose 2^-57 of it each (19 of them).
The global sums are plain FP64 sums of those (N terms, 2^-52 each way: N 2^-52 is far above what is seen).
"""
from fractions import Fraction

import numpy as np
import pytest
import torch

import paper_1410_0412_gb300 as lbm
from oracle.d3q19 import C, W

pytestmark = pytest.mark.gpu


def _grids(prec, shifted, n):
    rng = np.random.default_rng(8)
    w = np.asarray(W)[:, None]
    base = 0.0 if shifted else 1.0
    near = base * w * (1 + 0.01 * rng.standard_normal((19, n))) + (0.01 * w * rng.standard_normal((19, n)) if shifted else 0)
    out = [near, base * w + np.zeros((19, n)), base * w + 1e-7 * w * rng.standard_normal((19, n)),
           near * 2.0 ** rng.integers(-12, 3, (19, n)), base * w + (2.0 ** -140 if prec == "f32" else 2.0 ** -12) *
           rng.integers(-3, 4, (19, n)) * (1.0 if shifted else 0.0)]
    bad = near.copy()
    bad[3, 1::7] = np.inf
    bad[5, 2::7] = np.nan
    bad[:, 3::7] = -0.5
    bad[:, 4::7] = 0.0
    return out, bad


@pytest.mark.parametrize("prec,shifted", [("f64", False), ("f64", True), ("f32", False), ("f32", True), ("f16s", True)])
@pytest.mark.parametrize("g,drag", [((0.0, 0.0, 0.0), False), ((1e-6, 0.0, 0.0), True), ((1e-5, -3e-6, 2e-7), False)])
@pytest.mark.parametrize("X", [7, 100])
def test_readback_against_exact_sums(prec, shifted, g, drag, X):
    lat = lbm.Lattice(np.zeros((5, 6, X), np.uint8), periodic=(1, 1, 1)).upload()
    n = lat.N
    p = lbm.Params(g=g, shifted=shifted)
    s = np.linspace(0.0, 1.0, n, dtype=np.float32) if drag else None
    s_dev = torch.as_tensor(s, device="cuda") if drag else None
    grids, bad = _grids(prec, shifted, n)
    for grid in grids + [bad]:
        t = lat.new_grid(prec)
        scale = 1024.0 if prec == "f16s" else 1.0
        t[:, :n] = torch.as_tensor(grid * scale, device="cuda").to(t.dtype)
        d = t[:, :n].double().cpu().numpy() / scale
        rho, u, sums = (v.cpu().numpy() for v in lbm.lbm_macroscopic(lat, prec, p, t, lbm.LBM_LAYOUT_AA_EVEN, s_dev))
        F = lbm.lbm_canonical_pdfs(lat, prec, p, t, lbm.LBM_LAYOUT_AA_EVEN).cpu().numpy()
        want = d + np.asarray(W)[:, None] if shifted else d
        assert np.array_equal(F, want, equal_nan=True)
        for k in range(0, n, 3):
            if not np.isfinite(d[:, k]).all():
                assert not np.isfinite(rho[k]) and not np.isfinite(u[1, k])  # the Inf is in the +y PDF
                continue
            f = [Fraction(float(v)) for v in d[:, k]]
            r = sum(f) + (1 if shifted else 0)
            j = [sum(int(C[i][a]) * f[i] for i in range(19)) for a in range(3)]
            size = sum(abs(v) for v in f) + (1 if shifted else 0)
            cut = 19 * max(abs(v) for v in f) / 2 ** 57
            # a density that cancels (or is negative) takes the FP64 sums: their bound is in the terms' size
            slack = size * 19 / 2 ** 52 if r <= 0 or r < size / 4 else 0
            assert abs(Fraction(float(rho[k])) - r) <= r / 2 ** 52 + cut + slack
            if r <= 0 or r < size / 4:
                continue
            kd = 1 / (1 + Fraction(float(s[k])) / 2) if drag else Fraction(1)
            for a in range(3):
                ex = (j[a] / r + Fraction(g[a]) / 2) * kd
                tol = (abs(j[a]) / r + abs(Fraction(g[a]))) / 2 ** 50 + 2 * cut / r
                assert abs(Fraction(float(u[a, k])) - ex) <= tol, (k, a)
        if np.isfinite(rho).all() and np.isfinite(u).all():
            ref = [rho.sum()] + [(rho * u[a]).sum() for a in range(3)]
            mag = [np.abs(rho).sum()] + [np.abs(rho * u[a]).sum() for a in range(3)]
            assert all(abs(x - y) <= n * 2.0 ** -52 * m + 1e-300 for x, y, m in zip(sums, ref, mag))
