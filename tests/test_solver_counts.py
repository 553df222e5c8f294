"""Step counts that Solver.step takes in OS-NT form: none, odd, and more than 32 bits hold (no GPU: the call is faked)."""
import pytest

import paper_1410_0412_gb300 as lbm


@pytest.mark.parametrize("n", [-3, 0, 1, 2, 7, (1 << 30) - 1, 1 << 30, (1 << 30) + 1, (1 << 31) + 5, (1 << 33) + 4])
def test_osnt_counts(monkeypatch, n):
    calls = []

    def run(lat, prec, params, grid0, grid1, steps, s, ria, stream):
        assert 0 < steps < 1 << 31
        calls.append((grid0, grid1, steps))

    monkeypatch.setattr(lbm, "lbm_run_osnt", run)
    sim = object.__new__(lbm.Solver)
    sim.form, sim.lat, sim.prec, sim.params, sim.s, sim.ria, sim.t = "osnt", None, 0, None, None, True, 10
    sim.grids = ["a", "b"]
    sim.step(n)
    done = max(n, 0)
    assert sim.t == 10 + done and sum(c[2] for c in calls) == done
    assert sim.grids == (["b", "a"] if done % 2 else ["a", "b"])
    at = "a"
    for g0, g1, k in calls:  # each call starts from the grid that holds the state
        assert g0 == at and g1 != at
        at = g1 if k % 2 else g0
