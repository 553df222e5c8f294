"""FP64 collision of deviation storage where large deviations cancel in density and momentum.

A node under shear holds deviations whose density and momentum are far smaller than its largest member; with l+ = 1
its result follows from those two alone.  The fixed-point scale is tied to the largest deviation, so such nodes have
to take the FP64 update.  What the fixed-point route accepts has |S| >= 2^56 or |J| >= 2^57 units, hence an output of
at least 2^56 / 19 or (with the drag's factor of a third) 2^57 / 30 units, and at most 56 units of error: 2^-45 of the
largest output.  The FP64 update's dozen roundings are within 2^-48 of it, terms that cancel among the outputs aside.
"""
from fractions import Fraction

import numpy as np
import pytest
import torch

import paper_1410_0412_gb300 as lbm
from test_fx_collide import _exact


def _shear(n, seed):
    """Deviations of pure stress modes (exact zero density and momentum), plus a small momentum and density."""
    rng = np.random.default_rng(seed)
    d = np.zeros((n, 19))
    for k, (p, q) in enumerate([(1, 3), (3, 5), (7, 9), (11, 13), (15, 17)]):  # pairs of equal weight, opposite sign
        a = np.ldexp(rng.integers(-(1 << 20), 1 << 20, n).astype(float), -30)
        for i, v in ((p, a), (p + 1, a), (q, -a), (q + 1, -a)):
            d[:, i] += v
    small = np.ldexp(1.0, -rng.integers(15, 45, (n, 3)))
    for a in range(3):
        d[:, 2 * a + 1] += small[:, a] * (rng.random(n) < 0.7)
    return d


@pytest.mark.parametrize("omega", [1.0, 0.9999])
@pytest.mark.parametrize("drag", [False, True])
def test_cancelling_deviations_are_right_or_refused(omega, drag):
    p = lbm.Params(omega_plus=omega, magic=3 / 16, g=(0.0, 0.0, 0.0), rho0=1.0, shifted=True)
    d = _shear(200, 6)
    s = np.linspace(0.0, 1.0, 200, dtype=np.float32) if drag else None
    out, ok = lbm.lbm_fx_collide_host(d, p, s)
    for n in np.nonzero(ok)[0]:
        ex, _ = _exact(d[n], p, 0.0 if s is None else s[n])
        top = max(abs(v) for v in ex)
        assert max(abs(Fraction(float(out[n, i])) - ex[i]) for i in range(19)) <= top / 2 ** 45, n
    assert not ok.all()


def test_states_of_a_flow_stay_in_the_range():
    # at rest, under the force alone, density waves and flows keep to the fixed-point route
    from test_fx_collide import W, _nodes
    for g in ((0.0, 0.0, 0.0), (1e-6, 0.0, 0.0)):
        p = lbm.Params(g=g, rho0=1.0, shifted=True)
        for d in (np.zeros((4, 19)), np.outer([1e-9, -1e-3, 0.02], W), 1e-16 * np.outer([1, -1], W),
                  _nodes(300, 1, True, noise=2e-3, umax=0.02), _nodes(300, 2, True, noise=1e-4, umax=1e-3)):
            assert lbm.lbm_fx_collide_host(d, p)[1].all()


@pytest.mark.gpu
@pytest.mark.parametrize("drag", [False, True])
def test_step_of_cancelling_deviations(drag):
    lat = lbm.Lattice(np.zeros((3, 5, 13), np.uint8), periodic=(1, 1, 1)).upload()
    n = lat.N
    p = lbm.Params(omega_plus=1.0, magic=3 / 16, g=(0.0, 0.0, 0.0), rho0=1.0, shifted=True)
    d = _shear(n, 7)
    s = np.linspace(0.0, 1.0, n, dtype=np.float32) if drag else None
    grid = lat.new_grid("f64")
    grid[:, :n] = torch.as_tensor(d.T.copy(), device="cuda")
    lbm.lbm_step_aa(lat, "f64", p, grid, 0, torch.as_tensor(s, device="cuda") if drag else None)
    inv = [0] + [i + 1 if i % 2 else i - 1 for i in range(1, 19)]
    got = grid[inv, :n].cpu().numpy()
    for k in range(n):
        ex, _ = _exact(d[k], p, 0.0 if s is None else s[k])
        top = max(abs(v) for v in ex)
        assert max(abs(Fraction(float(got[i, k])) - ex[i]) for i in range(19)) <= top / 2 ** 45, k
