"""Finite positions beyond 2^53 cells (a run that has blown up passes through
them): their cell has to stay inside the grid - the fused remainder of the wrap
can lie anywhere - and the other particles' sets and fits are not touched."""
import numpy as np
import pytest

import oracle
import workloads
from _gpu import need_gpu, sets_of, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("which", ["lattice", "tube"])
def test_far_positions(which):
    phb = need_gpu()
    w = workloads.random_modes(12, seed=81) if which == "lattice" else workloads.shock_tube(9000, seed=81)
    far = np.array([5, 9, 100, 101, 1500])
    pos = w.pos.copy()
    pos[0, 5] = 1e30
    pos[:, 9] = (1e17, -3e200, 1e300)
    pos[2, 100] = -1e300
    pos[1, 101] = 2.2e25
    pos[:, 1500] = -7.7e18
    plan = phb.Plan.for_workload(w)
    lam, U = torch.tensor(w.lam, device="cuda"), torch.tensor(w.U, device="cuda")
    p = torch.tensor(pos, device="cuda")
    phb.build_neighbors(plan, p, lam)
    got = sets_of(*phb.export_neighbors(plan))
    off, idx = oracle.neighbors(oracle.box_of(w), w.pos, w.lam)
    for i in np.setdiff1d(np.arange(w.n), far):
        exp = idx[off[i]:off[i + 1]]
        np.testing.assert_array_equal(np.setdiff1d(got[i], far), np.setdiff1d(exp, far))
    for prec in ("fp32_mixed", "fp64"):
        phb.mhd_rhs(plan, phb.Params(gamma=w.gamma, precision=prec), p, lam, U)
        assert isinstance(plan.read_status(), int)


def test_position_lost_after_the_build():
    """A neighbour whose position is not a number when the fit runs is left out,
    in both precisions."""
    phb = need_gpu()
    w = workloads.random_modes(10, seed=82, amp=0.05)
    plan = phb.Plan.for_workload(w)
    pos, lam, U = phb.tensors_of(w)
    phb.build_neighbors(plan, pos, lam)
    for value in (float("nan"), -float("nan")):
        moved = pos.clone()
        moved[0, 17] = value
        out, _ = phb.mhd_rhs(plan, phb.Params(gamma=w.gamma, precision="fp64"), moved, lam, U)
        assert bool(torch.isfinite(out).all())
