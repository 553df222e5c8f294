"""The FP64 fixed-point routines at relaxation rates next to 0 and 2 (no GPU, and the steps on a GPU).

(1 - l+-)/2, l+/4 and a+/2 are factors of a product that holds fractions below 1/2 - 2^-33.  Rates beyond that have to
be refused (the kernels then take the FP64 update); accepted ones keep the bounds of the general tests.
"""
import numpy as np
import pytest
import torch

import paper_1410_0412_gb300 as lbm
import test_fx_adjoint
import test_fx_collide
from oracle import lbm as olbm
from oracle import tables as otables

RATES = [1e-12, 2e-11, 1e-10, 2e-10, 2.0 ** -32, 3e-10, 1e-9]


@pytest.mark.parametrize("shifted", [False, True])
@pytest.mark.parametrize("low", [True, False])
@pytest.mark.parametrize("rate", RATES)
@pytest.mark.parametrize("drag", [False, True])
def test_rates_at_the_ends_are_right_or_refused(shifted, low, rate, drag):
    p = lbm.Params(omega_plus=rate if low else 2 - rate, magic=3 / 16, g=(1e-6, 0.0, 0.0), rho0=1.0, shifted=shifted)
    s = np.linspace(0.0, 1.0, 12, dtype=np.float32) if drag else None
    ok = test_fx_collide._check(test_fx_collide._nodes(12, 5, shifted), p, s)
    d = test_fx_adjoint._forward(12, 4, shifted, 0.05)
    ok_adj = test_fx_adjoint._check(d, np.random.default_rng(3).standard_normal((12, 19)), p, s)
    if rate < 2e-10:
        assert not ok.any() and not ok_adj.any()
    if rate == 1e-9:
        assert ok.all() and ok_adj.all()


def test_pair_update_refuses_rates_it_cannot_hold():
    d, terms = np.tile(1 / 36 + np.arange(19) * 1e-4, (1, 1)), np.full((1, 10), 1e-3)
    for q, held in ((0.5 - 2.0 ** -53, False), (0.5 - 2.0 ** -34, False), (0.5 - 2.0 ** -32, True), (0.3, True)):
        for qm, qp, lp1 in ((q, 0.0, True), (-q, 0.0, True), (0.1, q, False), (0.1, -q, False)):
            out, ok = lbm.lbm_fx_pairs_host(d, terms, qm, qp, lp1)
            assert ok[0] == held
            if held:  # the pair's sum is 2 e, which qm does not enter; its difference is 2 o
                e = 2 * (1e-3 + 1e-6) + 2 * qp * (d[0, 1] + d[0, 2])
                o = 2 * qm * (d[0, 1] - d[0, 2]) + 2e-3
                assert abs(out[0, 1] + out[0, 2] - e) < 1e-15 and abs(out[0, 1] - out[0, 2] - o) < 1e-15


@pytest.mark.gpu
@pytest.mark.parametrize("form", ["aa", "osnt"])
@pytest.mark.parametrize("omega", [1e-12, 1e-10, 1e-9, 2 - 1e-9, 2 - 1e-10])
def test_steps_at_the_ends_of_the_rates(form, omega):
    solid = np.zeros((6, 7, 9), np.uint8)
    solid[2:4, 3, 4:6] = 1
    kw = dict(omega_plus=omega, magic=3 / 16, g=(1e-6, 0.0, 0.0))
    T, op = otables.Tables(solid, periodic=(1, 1, 1)), olbm.Params(**kw)
    gen = torch.Generator().manual_seed(5)
    F0 = olbm.uniform_state(T.N, op, 1.0, (0.01, -0.02, 0.005))
    F0 = F0 * (1 + 1e-2 * (torch.rand(F0.shape, generator=gen, dtype=torch.float64) - 0.5))
    layout, steps = (0, 4) if form == "osnt" else (1, 4)
    G = olbm.from_canonical(F0, layout, T.adj, op)
    G = olbm.run_osnt(G, T.adj, op, steps, None) if form == "osnt" else olbm.run_aa(G, T.adj, op, steps, 0, None)
    ref = olbm.canonical(G, layout, T.adj, op)
    for shifted in (False, True):
        sim = lbm.Solver(lbm.Lattice(solid, periodic=(1, 1, 1)).upload(), "f64", lbm.Params(shifted=shifted, **kw),
                         form=form, ria=True)
        sim.load(F0.cuda())
        sim.step(steps)
        assert float((sim.canonical().cpu() - ref).abs().max() / ref.abs().max()) <= 1e-12
