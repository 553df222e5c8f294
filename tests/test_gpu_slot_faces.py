"""Run slot tables of lattices with pressure faces, against the adjacency list, on a GPU.

A lattice with pressure faces and long runs steps through the run slot table, whose rows also hold the directions
that meet an inlet or an outlet; the adjacency list decodes the markers entry by entry.  Both evaluate the same
arithmetic, so the states after a few steps agree to the rounding of one operation per step and PDF: 8 steps at
2^-52, 2^-23 or 2^-10 of the largest PDF (the largest deviation in shifted storage).  The sizes put the last node at
the edges of a CTA; one lattice carries markers in every direction, as a caller's own adjacency list may.
"""
import numpy as np
import pytest
import torch

import paper_1410_0412_gb300 as lbm
from oracle import lbm as olbm

pytestmark = pytest.mark.gpu

EPS = {"f64": 2.0 ** -52, "f64df": 2.0 ** -44, "f32": 2.0 ** -23, "f16s": 2.0 ** -10}


def _lattice(kind, X):
    rng = np.random.default_rng(4)
    if kind == "duct":  # one row per (y, z): three runs a row, a solid voxel here and there
        solid = np.zeros((2, 3, X), np.uint8)
        solid[1, 1, X // 2] = 1
        return lbm.Lattice(solid, periodic=(0, 1, 1), x_pressure=True)
    # a caller's adjacency list: walls, inlets and outlets in every direction on some nodes
    base = lbm.Lattice(np.zeros((2, 3, X), np.uint8), periodic=(1, 1, 1))
    adj = base.tables()["adj"].copy()
    inv = [i + 1 if i % 2 else i - 1 for i in range(1, 19)]
    for n in rng.integers(0, base.N, max(2, base.N // 40)):
        i = int(rng.integers(1, 19))
        m = adj[i - 1, n]
        if m >= 0:  # cut the link on both sides
            adj[i - 1, n] = -int(rng.integers(1, 4))
            adj[inv[i - 1] - 1, m] = -int(rng.integers(1, 4))
    return lbm.Lattice.from_adjacency(adj)


@pytest.mark.parametrize("kind", ["duct", "raw"])
@pytest.mark.parametrize("X", [21, 22, 43, 85])  # 6 X - 1 or 6 X nodes: 125/126, 131/132, 257/258, 509/510
@pytest.mark.parametrize("prec", ["f64", "f64df", "f32", "f16s"])
@pytest.mark.parametrize("form", ["aa", "osnt"])
def test_slot_steps_match_adjacency_steps(kind, X, prec, form):
    lat = _lattice(kind, X)
    if not 2 * lat.R <= lat.N:
        pytest.skip("no slot table at this run count")
    lat.upload()
    p = lbm.Params(omega_plus=1.2, g=(1e-4, 0.0, -2e-5), shifted=prec in ("f32", "f16s"), rho_in=1.01, rho_out=0.99)
    op = olbm.Params(omega_plus=1.2, magic=3 / 16, g=p.g)
    gen = torch.Generator().manual_seed(2)
    F = olbm.uniform_state(lat.N, op, 1.0, (0.02, -0.01, 0.0))
    F = (F * (1 + 1e-2 * (torch.rand(F.shape, generator=gen, dtype=torch.float64) - 0.5))).cuda()
    s = torch.linspace(0, 0.5, lat.N).cuda()
    got = []
    for ria in (True, False):
        sim = lbm.Solver(lat, prec, p, form=form, ria=ria, s=s)
        sim.load(F)
        sim.step(8)
        got.append(sim.pdf.double()[:, :lat.N])
    top = got[1].abs().max()
    assert float((got[0] - got[1]).abs().max()) <= 8 * EPS[prec] * float(top)


@pytest.mark.parametrize("kind", ["duct", "raw"])
@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_adjoint_with_faces_matches_adjacency(kind, prec):
    lat = _lattice(kind, 43).upload()
    p = lbm.Params(g=(1e-4, 0.0, 0.0), shifted=True, rho_in=1.01, rho_out=0.99)
    G0 = lat.new_grid(prec)
    lbm.lbm_init_equilibrium(lat, prec, p, G0, lbm.LBM_LAYOUT_OSNT, 1.0, (0.01, 0.0, 0.0))
    grads = []
    for ria in (True, False):
        s = torch.linspace(0, 0.5, lat.N, device="cuda", dtype=torch.float64).requires_grad_(True)
        J = lbm.flux_objective(s, lat, prec, p, G0, 6, 3, ria)
        grads.append((float(J.detach()), torch.autograd.grad(J, s)[0]))
    eps = 6 * 8 * EPS[prec]
    assert abs(grads[0][0] - grads[1][0]) <= eps * abs(grads[1][0]) * 8
    assert float((grads[0][1] - grads[1][1]).abs().max()) <= eps * float(grads[1][1].abs().max())
