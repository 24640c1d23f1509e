"""Tiles that hold particles without a finite position, which are in no cell:
their slots have no staged record of their own."""
import numpy as np
import pytest

import oracle
import workloads
from _gpu import need_gpu, rhs_err, rhs_term_scales, sets_of, torch

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


def lattice(seed):
    """A lattice in storage order, and its lists' oracle."""
    phb = need_gpu()
    w = workloads.random_modes(12, seed=seed, amp=0.05)
    plan = phb.Plan.for_workload(w)
    pos, lam, U = phb.tensors_of(w)
    phb.build_neighbors(plan, pos, lam)
    phb.reorder(plan, pos, lam, U)
    w.pos, w.lam, w.U = pos.cpu().numpy(), lam.cpu().numpy(), U.cpu().numpy()
    phb.build_neighbors(plan, pos, lam)
    return phb, w, plan, pos, lam, U


def without(w, lost):
    """Right-hand sides and their term scales from lists that leave `lost` out."""
    box = oracle.box_of(w)
    off, idx = oracle.neighbors(box, w.pos, w.lam)
    keep = ~np.isin(idx, lost)
    cut = np.concatenate([[0], np.cumsum(keep)])[off]
    nb = (cut.astype(off.dtype), idx[keep])
    exp, st = oracle.mhd_rhs(box, w.pos, w.lam, w.U, nb, gamma=w.gamma)
    g, h, _ = oracle.mls_derivs(box, w.pos, w.lam, w.U, nb, gamma=w.gamma)
    assert not st.any()
    return exp, rhs_term_scales(w.U, g, h, w.gamma)


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("value", [np.nan, -np.nan, np.inf])
@pytest.mark.parametrize("slot", ["first", "middle"])
def test_position_lost_after_the_build(axis, value, slot):
    """A neighbour whose position is not a number or infinite when the fit
    runs is left out of every fit that lists it, in both precisions."""
    phb, w, plan, pos, lam, U = lattice(82)
    lost = 128 * 3 + {"first": 0, "middle": 64}[slot]   # a tile is staged relative to its middle slot
    exp, sc = without(w, [lost])
    other = np.setdiff1d(np.arange(w.n), [lost])
    pos[axis, lost] = value
    for prec, tol in (("fp64", 1e-12), ("fp32_mixed", 1e-5)):
        out, _ = phb.mhd_rhs(plan, phb.Params(gamma=w.gamma, precision=prec), pos, lam, U)
        e = rhs_err(out.cpu().numpy()[:, other], exp[:, other], sc)
        assert e.max() < tol, (prec, e)


@pytest.mark.parametrize("value", [np.nan, np.inf])
@pytest.mark.parametrize("field", [0, 3, 7])
def test_field_lost(field, value):
    """A field that is not finite, of a tile's middle particle, reaches the
    particles that list it and no others."""
    phb, w, plan, pos, lam, U = lattice(83)
    lost = 128 * 5 + 64
    exp, sc = without(w, [])
    got = sets_of(*phb.export_neighbors(plan))
    far = np.array([i for i in range(w.n) if i != lost and lost not in got[i]])
    assert 32 < w.n - far.size < 80
    U[field, lost] = value
    for prec, tol in (("fp64", 1e-12), ("fp32_mixed", 1e-5)):
        out, _ = phb.mhd_rhs(plan, phb.Params(gamma=w.gamma, precision=prec), pos, lam, U)
        e = rhs_err(out.cpu().numpy()[:, far], exp[:, far], sc)
        assert e.max() < tol, (prec, e)


@pytest.mark.parametrize("side", [12, 26])
def test_positions_far_away_before_the_build(side):
    """Finite positions beyond 2^53 cells are counted to an edge cell, whose tile
    they must not spoil: fits of the particles that do not list one are those of
    the set without them, in both precisions.  (Sets of both searches.)"""
    phb = need_gpu()
    w = workloads.random_modes(side, seed=84, amp=0.05)
    rng = np.random.default_rng(9)
    # the caller's first particles lie about the cells that far positions are counted to
    lost = np.concatenate([np.arange(0, 60, 2), rng.permutation(w.n)[:30]])
    exp, sc = without(w, lost)
    pos, lam, U = (torch.tensor(x, device="cuda") for x in (w.pos, w.lam, w.U))
    at = torch.tensor(lost, device="cuda")
    pos[:, at] = torch.tensor(rng.choice([1e30, -3e200, 1e300, 2.2e25, -7.7e18], (3, lost.size)), device="cuda")
    plan = phb.Plan.for_workload(w)
    phb.build_neighbors(plan, pos, lam, check_capacity=False)
    got = sets_of(*phb.export_neighbors(plan))
    is_lost = np.zeros(w.n, bool)
    is_lost[lost] = True
    far = np.array([i for i in range(w.n) if not is_lost[i] and not is_lost[got[i]].any()])
    assert far.size > w.n // 2
    for prec, tol in (("fp64", 1e-12), ("fp32_mixed", 1e-5)):
        out, _ = phb.mhd_rhs(plan, phb.Params(gamma=w.gamma, precision=prec), pos, lam, U)
        e = rhs_err(out.cpu().numpy()[:, far], exp[:, far], sc)
        assert e.max() < tol, (prec, e)
