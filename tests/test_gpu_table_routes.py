"""The tables that the steps choose by order and size, against each other, on a GPU.

On a Hilbert curve (about one run per node, more than 2^18 nodes) the single-precision AA odd steps read adjacency
entries where row order reads resolved slots; large FP32 AA and FP16S OS-NT steps with the adjacency list read entries
too.  All evaluate the same arithmetic, so the states after a few steps agree to the rounding of one operation per
step and PDF: 5 steps at 2^-52, 2^-23 or 2^-10 of the largest stored value.
"""
import numpy as np
import pytest
import torch

import geometry
import paper_1410_0412_gb300 as lbm
from oracle import lbm as olbm

pytestmark = pytest.mark.gpu

EPS = {"f64": 2.0 ** -52, "f32": 2.0 ** -23, "f16s": 2.0 ** -10}


def _steps(lat, prec, form, ria, order, s):
    p = lbm.Params(omega_plus=1.2, g=(1e-4, 0.0, -2e-5), shifted=prec != "f64")
    gen = torch.Generator().manual_seed(2)
    F = olbm.uniform_state(lat.N, olbm.Params(), 1.0, (0.02, -0.01, 0.0))
    F = (F * (1 + 1e-2 * (torch.rand(F.shape, generator=gen, dtype=torch.float64) - 0.5))).cuda()
    sim = lbm.Solver(lat, prec, p, form=form, ria=ria, s=s[order].contiguous() if s is not None else None)
    sim.load(F[:, order].contiguous())
    sim.step(5)
    back = torch.empty_like(order)
    back[order] = torch.arange(lat.N, device="cuda")
    return sim.canonical()[:, back]


@pytest.mark.parametrize("prec", ["f64", "f32", "f16s"])
@pytest.mark.parametrize("form", ["aa", "osnt"])
@pytest.mark.parametrize("drag", [False, True])
def test_hilbert_order_matches_row_order(prec, form, drag):
    solid = geometry.random_voxels(73, 71, 69, 0.2, 5)
    solid[:, :, 73 - 60:] = 0  # long rows, so that row order has few runs
    lats = [lbm.Lattice(solid, periodic=(1, 0, 1), enum=e, B=1).upload() for e in ("lex", "hilbert")]
    n = lats[0].N
    assert n > 1 << 18 and 2 * lats[0].R <= n < 2 * lats[1].R
    key = [torch.as_tensor((l.tables()["node_xyz"].astype(np.int64) * [1, 128, 128 * 128]).sum(1)).cuda() for l in lats]
    order = torch.searchsorted(key[0].sort().values, key[1])
    assert (key[0].sort().values == key[0]).all()
    s = torch.linspace(0, 0.5, n).cuda() if drag else None
    ident = torch.arange(n, device="cuda")
    want = _steps(lats[0], prec, form, True, ident, s)
    w = torch.tensor([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12, dtype=torch.float64, device="cuda")[:, None]
    top = float((want - (w if prec != "f64" else 0)).abs().max())
    for lat, ria, o in ((lats[0], False, ident), (lats[1], True, order), (lats[1], False, order)):
        got = _steps(lat, prec, form, ria, o, s)
        assert float((got - want).abs().max()) <= 5 * EPS[prec] * top


@pytest.mark.parametrize("prec,form,side", [("f32", "aa", 123), ("f16s", "osnt", 155)])
def test_large_lists_match_runs(prec, form, side):
    lat = lbm.Lattice(np.zeros((side, side, side), np.uint8), periodic=(1, 1, 1)).upload()
    assert 38 * lat.N * (4 if prec == "f32" else 2) > 256 << 20 and 10 * lat.R < lat.N
    ident = torch.arange(lat.N, device="cuda")
    a, b = (_steps(lat, prec, form, ria, ident, None) for ria in (True, False))
    w = torch.tensor([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12, dtype=torch.float64, device="cuda")[:, None]
    assert float((a - b).abs().max()) <= 5 * EPS[prec] * float((a - w).abs().max())
