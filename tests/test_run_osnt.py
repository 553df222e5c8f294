"""lbm_run_osnt: several OS-NT steps in one call, and Solver.step / step_graph on top of it."""
import ctypes

import numpy as np
import pytest
import torch

import paper_1410_0412_gb300 as lbm
from paper_1410_0412_gb300 import _lib


def test_run_osnt_argument_checks():
    lat = lbm.Lattice(np.zeros((2, 2, 2), np.uint8), periodic=(1, 1, 1))
    lib, p = _lib.load(), lbm.Params().c()
    a, b = ctypes.c_void_p(4096), ctypes.c_void_p(8192)
    for g0, g1, steps in ((None, b, 1), (a, None, 1), (a, a, 1), (a, b, -1), (a, b, 1)):  # the last: no tables
        assert lib.lbm_run_osnt(lat.handle, 0, ctypes.byref(p), g0, g1, steps, None, 0, None) != 0
    assert lib.lbm_run_osnt(lat.handle, 0, ctypes.byref(p), a, b, 0, None, 0, None) == 0


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["f64", "f32", "f16s"])
@pytest.mark.parametrize("n", [0, 1, 2, 3, 8])
def test_run_osnt_equals_single_steps(prec, n):
    solid = np.zeros((6, 7, 23), np.uint8)
    solid[2:4, 3, 5:9] = 1
    lat = lbm.Lattice(solid, periodic=(1, 0, 1)).upload()
    p = lbm.Params(g=(1e-5, 0.0, 0.0), shifted=prec != "f64")
    sims = [lbm.Solver(lat, prec, p, form="osnt") for _ in range(2)]
    for sim in sims:
        sim.init_equilibrium(1.0, (0.02, 0.0, 0.0))
    sims[0].step(n)
    for _ in range(n):
        sim = sims[1]
        lbm.lbm_step_osnt(lat, prec, p, sim.grids[0], sim.grids[1], None, True)
        sim.grids.reverse()
    assert sims[0].t == n and torch.equal(sims[0].pdf, sims[1].pdf)


@pytest.mark.gpu
@pytest.mark.parametrize("form", ["aa", "osnt", "et"])
def test_step_graph_blocks_equal_steps(form):
    # 2 direct steps, then blocks of 16 pairs and single pairs, twice; the counts straddle the block length
    lat = lbm.Lattice(np.zeros((4, 5, 21), np.uint8), periodic=(1, 1, 1)).upload(
        lbm.LBM_TABLES_ADJ | lbm.LBM_TABLES_RIA | lbm.LBM_TABLES_ET)
    p = lbm.Params(g=(1e-5, 2e-6, 0.0))
    sims = [lbm.Solver(lat, "f64", p, form=form) for _ in range(2)]
    for sim in sims:
        sim.init_equilibrium(1.0, (0.02, 0.0, 0.0))
    for n in (2, 30, 32, 34, 70):
        sims[0].step_graph(n)
        sims[1].step(n)
        assert sims[0].t == sims[1].t and torch.equal(sims[0].pdf, sims[1].pdf)
