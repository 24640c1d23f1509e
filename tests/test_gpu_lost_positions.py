"""Tiles that hold particles without a finite position, which are in no cell:
their slots have no staged record of their own."""
import numpy as np
import pytest

import workloads
from _gpu import need_gpu, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("spare", [0, 1])
def test_lost_slots_of_a_full_stage(spare):
    """100 particles in the last cell before the periodic corner and 28 lost
    ones, in one tile: the cell that the lost slots are counted to, (0, 0, 0), is
    empty and comes after all staged records, which fill the stage.  The others
    get what they get without the lost ones, within the corrected fit's rounding
    (eps 6e-8 times sqrt(cond) <= 173, an order of magnitude for the sums)."""
    phb = need_gpu()
    rng = np.random.default_rng(21 + spare)
    n, m = 128, 100
    pos = rng.uniform(0.876, 0.999, (3, n))
    U = workloads.configs.background(n) + 0.05 * np.sin(8 * pos[np.arange(8) % 3] + np.arange(8)[:, None])
    lam = np.full(n, 0.05)
    lost = rng.permutation(n)[:n - m]
    keep = np.setdiff1d(np.arange(n), lost)
    bad = pos.copy()
    bad[1, lost] = np.nan

    def derivs(x, sel):
        w = workloads.Workload("lost", np.zeros(3), np.ones(3), np.ones(3, np.int32), x[:, sel].copy(),
                               lam[sel].copy(), U[:, sel].copy(), 5.0 / 3.0)
        plan = phb.Plan.for_workload(w, stage_cap=m + spare, nbr_capacity=n * n)
        assert list(plan.c.ncell) == [8, 8, 8]
        p, l, u = phb.tensors_of(w)
        phb.build_neighbors(plan, p, l, check_capacity=False)
        assert plan.stats()["build_fallback_tiles"] == 0
        g, _, st = phb.mls_derivs(plan, phb.Params(gamma=w.gamma, refine="on"), p, l, u)
        return g.cpu().numpy(), st.cpu().numpy()

    (g, st), (g0, st0) = derivs(bad, np.arange(n)), derivs(pos, keep)
    np.testing.assert_array_equal(st[keep] == 1, st0 == 1)
    assert (st0 != 1).sum() > 80
    assert np.abs(g[..., keep] - g0).max() <= 1e-4 * np.abs(g0).max()
    assert (st[lost] == 1).all() and not g[..., lost].any()
