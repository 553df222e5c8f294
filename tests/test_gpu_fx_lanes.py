"""The FP64 step gives a node in its fixed-point range the same bits whatever nodes share its warp, on a GPU.

The even AA step is local, so permuting the nodes of a grid must permute its result; the partitioned step regroups
nodes into other warps, so its chunks must reproduce the whole lattice.  The states mix nodes of every kind that is in
range (which the host image confirms): positive PDFs within 5 binades, a pair many binades below the others, a
negative pair, and, in deviation storage, deviations of one sign far below the force.
"""
import numpy as np
import pytest
import torch

import geometry
import paper_1410_0412_gb300 as lbm
from oracle import lbm as olbm

pytestmark = pytest.mark.gpu


def _mixed(n, seed, shifted):
    g = torch.Generator().manual_seed(seed)
    rnd = lambda *k: torch.rand(k, generator=g, dtype=torch.float64)
    F = olbm.uniform_state(n, olbm.Params(), 1.0, (0.01, -0.02, 0.005)) * (1 + 1e-2 * (rnd(19, n) - 0.5))
    kind = torch.randint(0, 100, (n,), generator=g)  # few, so that some warps hold none
    pair = torch.randint(1, 10, (n,), generator=g)  # one opposite pair, so that the velocity stays small
    hit = torch.stack([(torch.full((n,), (i + 1) // 2) == pair) for i in range(19)])
    F = torch.where(hit & (kind == 0), F * 2.0 ** -torch.randint(4, 14, (n,), generator=g).double(), F)
    F = torch.where(hit & (kind == 1), -0.3 * F, F)
    if shifted:
        w = torch.tensor([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12, dtype=torch.float64)[:, None]
        F = torch.where(kind == 2, w * (1 + 1e-13 * rnd(19, n)), F)
    return F


def _all_in_range(F, p, s=None):
    d = F.cpu().numpy().T - (np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12) if p.shifted else 0.0)
    return lbm.lbm_fx_collide_host(d, p, None if s is None else s.cpu().numpy())[1].all()


@pytest.mark.parametrize("omega", [1.0, 0.8])
@pytest.mark.parametrize("shifted", [False, True])
@pytest.mark.parametrize("drag", [False, True])
def test_even_step_commutes_with_permutations(omega, shifted, drag):
    lat = lbm.Lattice(np.zeros((17, 19, 23), np.uint8), periodic=(1, 1, 1)).upload()
    n = lat.N
    p = lbm.Params(omega_plus=omega, g=(1e-4, 2e-5, -3e-5), shifted=shifted)
    F = _mixed(n, 3, shifted).cuda()
    s = torch.linspace(0.0, 1.0, n).cuda() if drag else None
    assert _all_in_range(F, p, s)
    order = torch.randperm(n, generator=torch.Generator().manual_seed(8)).cuda()
    out = []
    for o in (torch.arange(n, device="cuda"), order):
        grid = lat.new_grid("f64")
        lbm.lbm_load_canonical(lat, "f64", p, F[:, o].contiguous(), grid, lbm.LBM_LAYOUT_AA_EVEN)
        lbm.lbm_step_aa(lat, "f64", p, grid, 0, s[o].contiguous() if drag else None)
        out.append(grid[:, :n].clone())
    assert torch.equal(out[0][:, order].view(torch.int64), out[1].view(torch.int64))


@pytest.mark.parametrize("shifted", [False, True])
@pytest.mark.parametrize("drag", [False, True])
def test_unit_rate_commutes_with_permutations_out_of_range_too(shifted, drag):
    lat = lbm.Lattice(np.zeros((17, 19, 23), np.uint8), periodic=(1, 1, 1)).upload()
    n = lat.N
    p = lbm.Params(omega_plus=1.0, g=(1e-4, 2e-5, -3e-5), shifted=shifted)
    F = _mixed(n, 3, shifted)
    kind = torch.randint(0, 60, (n,), generator=torch.Generator().manual_seed(1))
    F = torch.where(kind == 0, olbm.uniform_state(n, olbm.Params(), 1.0, (0.3, 0.1, 0.0)), F)
    F = torch.where(kind == 1, -F, F).cuda()
    s = torch.linspace(-0.01, 1.01, n).cuda() if drag else None
    order = torch.randperm(n, generator=torch.Generator().manual_seed(8)).cuda()
    out = []
    for o in (torch.arange(n, device="cuda"), order):
        grid = lat.new_grid("f64")
        lbm.lbm_load_canonical(lat, "f64", p, F[:, o].contiguous(), grid, lbm.LBM_LAYOUT_AA_EVEN)
        lbm.lbm_step_aa(lat, "f64", p, grid, 0, s[o].contiguous() if drag else None)
        out.append(grid[:, :n].clone())
    assert torch.isfinite(out[0]).all()
    assert torch.equal(out[0][:, order].view(torch.int64), out[1].view(torch.int64))


@pytest.mark.parametrize("form", ["osnt", "aa"])
@pytest.mark.parametrize("ria", [False, True])
@pytest.mark.parametrize("shifted", [False, True])
def test_partitioned_equals_whole_at_unit_rate(form, ria, shifted):
    solid = geometry.random_voxels(29, 23, 19, 0.25, 70)
    lat = lbm.Lattice(solid, periodic=(1, 0, 0)).upload()
    part = lbm.Partitioning(lat, 7).upload()
    p = lbm.Params(omega_plus=1.0, g=(1e-4, 2e-5, -3e-5), shifted=shifted)
    whole = lbm.Solver(lat, "f64", p, form=form, ria=ria)
    whole.load(_mixed(lat.N, 5, shifted).cuda())
    chunks = lbm.PartitionedSolver(part, "f64", p, form=form, ria=ria)
    chunks.load_global(whole.pdf)
    for _ in range(4):
        whole.step(1)
        chunks.step(1)
        assert torch.equal(chunks.to_global().view(torch.int64), whole.pdf[:, :lat.N].view(torch.int64))


@pytest.mark.parametrize("form", ["osnt", "aa"])
@pytest.mark.parametrize("ria", [False, True])
@pytest.mark.parametrize("prec", ["f64", "f32", "f16s"])
def test_chunks_equal_a_whole_that_steps_by_other_tables(form, ria, prec):
    # 345 k nodes on a Hilbert curve: the whole lattice is past the size where the tables change, its chunks are not
    solid = geometry.random_voxels(73, 71, 69, 0.05, 5)
    lat = lbm.Lattice(solid, periodic=(1, 0, 1), enum="hilbert").upload()
    assert lat.N > 1 << 18
    part = lbm.Partitioning(lat, 3).upload()
    p = lbm.Params(omega_plus=1.0, g=(1e-4, 2e-5, -3e-5), shifted=prec != "f64")
    whole = lbm.Solver(lat, prec, p, form=form, ria=ria)
    whole.load(_mixed(lat.N, 5, False).cuda())
    chunks = lbm.PartitionedSolver(part, prec, p, form=form, ria=ria)
    chunks.load_global(whole.pdf)
    it = {"f64": torch.int64, "f32": torch.int32, "f16s": torch.int16}[prec]
    for _ in range(3):
        whole.step(1)
        chunks.step(1)
        assert torch.equal(chunks.to_global().view(it), whole.pdf[:, :lat.N].view(it))
