"""The corrected step's reads of the neighbour lists: one entry at a time (queue)
and in aligned pairs (inside the tiles), over lists that start and end on odd
entries, of fewer entries than are read ahead, and whose last one ends at the
list region's capacity."""
import numpy as np
import pytest

import workloads
from _gpu import need_gpu, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [129, 2000, 4097])
@pytest.mark.parametrize("more", [0, 1])
def test_pairs_and_single_entries_agree(n, more):
    """Bit-identical, by construction: the same arithmetic on the same records."""
    phb = need_gpu()
    rng = np.random.default_rng(n)
    side = (n / 2000) ** (1 / 3)
    U = workloads.configs.background(n)
    U[0] *= 1 + 0.1 * rng.uniform(-1, 1, n)
    U[1:4] += 0.1 * rng.uniform(-1, 1, (3, n))
    w = workloads.Workload("lists", np.zeros(3), np.full(3, 1.0), np.zeros(3, np.int32),
                           side * rng.uniform(0, 1, (3, n)), rng.uniform(0.05, 0.11, n), U, 5.0 / 3.0)
    pos, lam, Ut = phb.tensors_of(w)
    plan = phb.Plan.for_workload(w)
    phb.build_neighbors(plan, pos, lam)
    total = plan.neighbor_total()
    plan = phb.Plan.for_workload(w, nbr_capacity=total + more)   # `more` of the two makes it odd
    phb.build_neighbors(plan, pos, lam)
    assert plan.c.nbr_capacity == total + more
    out = []
    for sched in ("queue", "tile"):
        prm = phb.Params(gamma=w.gamma, refine="on", refine_schedule=sched)
        out.append(phb.mhd_rhs(plan, prm, pos, lam, Ut)[0].clone())
        assert plan.stats()["refined_tiles"] > 0
    assert torch.equal(out[0], out[1])


@pytest.mark.parametrize("n,active", [(65_535, 0), (65_536, 0), (131_100, 65_535), (131_100, 65_536)])
def test_either_side_of_the_queue(n, active):
    """The default schedule on both sides of 65,536 fits, of a whole set and of an
    active subset by listed slots, against both forced ones, bit for bit."""
    phb = need_gpu()
    w = workloads.shear_layer(n, seed=5)
    n = w.n
    pos, lam, Ut = phb.tensors_of(w)
    plan = phb.Plan.for_workload(w)
    phb.build_neighbors(plan, pos, lam)
    idx = torch.tensor(np.random.default_rng(7).permutation(n)[:active].astype(np.int32), device="cuda")
    out = []
    for sched in ("auto", "queue", "tile"):
        prm = phb.Params(gamma=w.gamma, refine="on", refine_schedule=sched)
        if active:
            out.append(phb.mhd_rhs_active(plan, prm, pos, lam, Ut, idx).clone())
        else:
            out.append(phb.mhd_rhs(plan, prm, pos, lam, Ut)[0].clone())
        assert plan.stats()["refined_tiles"] > 0
    assert torch.equal(out[0], out[1]) and torch.equal(out[0], out[2])
