"""Particles whose lambda lies outside the plan's range (reported by the build's
status word): a lambda without a reach - infinite, negative, not a number or
beyond 2^30 cells - has no neighbours, one whose reach exceeds the box has them
all, and the other particles' sets and fits are those of the set without it."""
import numpy as np
import pytest

import workloads
from _gpu import need_gpu, sets_of, torch

pytestmark = pytest.mark.gpu

BAD = (np.inf, -np.inf, 1e300, -1e300, -5.0, -0.4, np.nan, 0.0, 3e11)


@pytest.mark.parametrize("periodic", [(1, 1, 1), (0, 1, 0)])
@pytest.mark.parametrize("which", ["one, small", "one, by cells", "varying", "varying, by threads"])
def test_lambda_without_a_reach(which, periodic):
    phb = need_gpu()
    w = {"one, small": lambda: workloads.random_modes(10, seed=3), "one, by cells": lambda: workloads.random_modes(26, seed=3),
         "varying": lambda: workloads.shock_tube(6000, seed=3),
         "varying, by threads": lambda: workloads.shock_tube((1 << 17) + 1000, seed=3)}[which]()
    w.periodic[:] = periodic
    n = w.n
    rng = np.random.default_rng(5)
    at = rng.permutation(n)[:len(BAD)]
    plan = phb.Plan.for_workload(w)
    pos, lam, U = phb.tensors_of(w)
    prm = phb.Params(gamma=w.gamma, precision="fp64")
    phb.build_neighbors(plan, pos, lam)
    exp = sets_of(*phb.export_neighbors(plan))
    ref, _ = phb.mhd_rhs(plan, prm, pos, lam, U)
    lam[torch.tensor(at, device="cuda")] = torch.tensor(BAD, dtype=torch.float64, device="cuda")
    with pytest.raises(phb.PhbError):
        phb.build_neighbors(plan, pos, lam)
    got = sets_of(*phb.export_neighbors(plan))
    other = np.setdiff1d(np.arange(n), at)
    for i in other[:: max(1, n // 3000)]:
        np.testing.assert_array_equal(got[i], exp[i])
    assert all(got[i].size == 0 for i in at)
    keep = torch.tensor(other, device="cuda")
    out, _ = phb.mhd_rhs(plan, prm, pos, lam, U)
    assert torch.equal(out[:, keep], ref[:, keep])
    mixed, _ = phb.mhd_rhs(plan, phb.Params(gamma=w.gamma), pos, lam, U)
    torch.cuda.synchronize()
    assert bool(torch.isfinite(mixed[:, keep]).all())


@pytest.mark.parametrize("periodic", [(1, 1, 1), (0, 0, 0)])
def test_reach_beyond_the_box(periodic):
    phb = need_gpu()
    w = workloads.random_modes(9, seed=4)
    w.periodic[:] = periodic
    n = w.n
    plan = phb.Plan.for_workload(w)
    pos, lam, _ = phb.tensors_of(w)
    lam[17] = 3.0
    lam[400] = 1e6
    with pytest.raises(phb.PhbError):
        phb.build_neighbors(plan, pos, lam)
    got = sets_of(*phb.export_neighbors(plan))
    for i in (17, 400):
        np.testing.assert_array_equal(got[i], np.setdiff1d(np.arange(n), [i]))
