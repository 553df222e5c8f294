"""Read-back of uniform flows whose velocity or momentum is a power of two, on each axis and in each storage.

Every node holds the same PDFs, so one exact rational value serves the whole grid.  Tolerance: rho is rounded once and
the quotient once, (1 + 2^-4) 2^-52 of |j / rho|, and FP64 PDFs more than 5 binades below the largest lose 2^-57 of it
each (19 of them); the global sums add N such terms in FP64.
"""
from fractions import Fraction

import numpy as np
import pytest
import torch

import paper_1410_0412_gb300 as lbm
from oracle.d3q19 import C, W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,shifted", [("f64", False), ("f64", True), ("f32", False), ("f32", True), ("f16s", True)])
def test_uniform_power_of_two_velocities_read_back(prec, shifted):
    lat = lbm.Lattice(np.zeros((3, 5, 9), np.uint8), periodic=(1, 1, 1)).upload()
    n, p = lat.N, lbm.Params(g=(0.0, 0.0, 0.0), shifted=shifted)
    scale = 1024.0 if prec == "f16s" else 1.0
    w, c = np.asarray(W, dtype=np.float64), np.asarray(C, dtype=np.float64)
    t = lat.new_grid(prec)
    for rho in (1.0, 1.01):
        for k in (3, 4, 5, 8):
            for v in (2.0 ** -k, -2.0 ** -k, 2.0 ** -k / rho, -2.0 ** -k / rho):
                for a in range(3):
                    u = np.zeros(3)
                    u[a] = v
                    cu = c @ u
                    d = w * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * (u @ u)) - (w if shifted else 0)
                    t[:, :n] = torch.as_tensor(d[:, None] * scale, device="cuda").to(t.dtype)
                    f = [Fraction(float(x)) for x in (t[:, 0].double() / scale).cpu().numpy()]
                    r = sum(f) + (1 if shifted else 0)
                    cut = 19 * max(abs(x) for x in f) / 2 ** 57
                    got, vel, sums = (x.cpu().numpy() for x in
                                      lbm.lbm_macroscopic(lat, prec, p, t, lbm.LBM_LAYOUT_AA_EVEN))
                    assert (got == got[0]).all() and abs(Fraction(float(got[0])) - r) <= r / 2 ** 52 + cut
                    for b in range(3):
                        ex = sum(int(C[i][b]) * f[i] for i in range(19)) / r
                        tol = abs(ex) * Fraction(17, 16) / 2 ** 52 + 2 * cut / r
                        assert (vel[b] == vel[b, 0]).all()
                        assert abs(Fraction(float(vel[b, 0])) - ex) <= tol, (rho, v, a, b)
                        assert abs(Fraction(float(sums[1 + b])) - n * r * ex) <= n * r * (tol + abs(ex) * n / 2 ** 52)
