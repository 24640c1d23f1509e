"""The adjoint's reverse lists at the lengths where their order comes about in
another way (a warp's registers up to 128 entries, sorted in place beyond) and
around powers of two."""
import numpy as np
import pytest

import oracle
import workloads
from _gpu import need_gpu, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [33, 128, 129, 130, 257, 258, 1000, 1025, 1026])
def test_everyone_names_everyone(n):
    """A ball of n particles within each other's r_f: each is named by n - 1
    lists.  <gbar, J v> of the oracle equals <J^T gbar, v>, and two calls agree
    bit for bit."""
    phb = need_gpu()
    rng = np.random.default_rng(n)
    x = rng.standard_normal((3, n))
    x *= rng.uniform(0, 1, n) ** (1 / 3) / np.linalg.norm(x, axis=0)   # the unit ball
    lam = np.full(n, 0.05)
    pos = 0.5 + 1.1 * lam * x   # at most 2.2 of r_f's 2.3 lambda apart
    U = workloads.configs.background(n) + 0.05 * np.sin(20 * pos[np.arange(8) % 3] + np.arange(8)[:, None])
    w = workloads.Workload("ball", np.zeros(3), np.ones(3), np.ones(3, np.int32), pos, lam, U, 5.0 / 3.0)
    plan = phb.Plan.for_workload(w, nbr_capacity=n * n)
    p, lam_t, u = phb.tensors_of(w)
    phb.build_neighbors(plan, p, lam_t)
    assert plan.neighbor_total() == n * (n - 1)
    prm = phb.Params(gamma=w.gamma, precision="fp64")
    gbar = rng.standard_normal((8, n))
    Ub, xb = phb.rhs_adjoint(plan, prm, p, lam_t, u, torch.tensor(gbar, device="cuda"))
    again = phb.rhs_adjoint(plan, prm, p, lam_t, u, torch.tensor(gbar, device="cuda"))
    assert torch.equal(Ub, again[0]) and torch.equal(xb, again[1])
    vpos, vU = rng.standard_normal((3, n)) * w.lam, rng.standard_normal((8, n))
    box = oracle.box_of(w)
    _, jv = oracle.rhs_jvp(box, w.pos, w.lam, w.U, vpos, vU, oracle.neighbors(box, w.pos, w.lam), gamma=w.gamma)
    lhs, rhs = float((gbar * jv).sum()), float((Ub.cpu().numpy() * vU).sum() + (xb.cpu().numpy() * vpos).sum())
    assert abs(lhs - rhs) <= 1e-10 * max(np.abs(gbar * jv).sum(), 1.0), (lhs, rhs)
