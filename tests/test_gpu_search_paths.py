"""Neighbour sets where the search changes path: one lambda below and above the
cell-major search's smallest set, reaches that cover a whole periodic axis,
open axes, lists longer than their scratch rows, cells of thousands of members
and particles without a finite position, against brute force; and the same
lists from every path."""
import numpy as np
import pytest

import oracle
import workloads
from _gpu import need_gpu, sample, sets_of, torch

pytestmark = pytest.mark.gpu


def sets(phb, w, **kw):
    plan = phb.Plan.for_workload(w, **kw)
    pos, lam, _ = phb.tensors_of(w)
    phb.build_neighbors(plan, pos, lam)
    return sets_of(*phb.export_neighbors(plan))


def check(w, got, query=None):
    q = np.arange(w.n) if query is None else query
    off, idx = oracle.neighbors(oracle.box_of(w), w.pos, w.lam, q)
    for k, i in enumerate(q):
        np.testing.assert_array_equal(got[i], idx[off[k]:off[k + 1]])


@pytest.mark.parametrize("side", [5, 25, 26])   # 15,625 and 17,576 particles
def test_one_lambda_either_side_of_the_cell_search(side):
    phb = need_gpu()
    w = workloads.random_modes(side, seed=side)
    check(w, sets(phb, w), None if side == 5 else sample(w.n, 400, seed=1))


@pytest.mark.parametrize("n", [40, 3000, 10_007])
@pytest.mark.parametrize("periodic", [(1, 1, 1), (0, 1, 0), (0, 0, 0)])
def test_varying_lambda(n, periodic):
    """10,007 shock-tube particles: coarse particles reach across y and z."""
    phb = need_gpu()
    rng = np.random.default_rng(n)
    w = workloads.shock_tube(n, seed=3) if n > 5000 else workloads.Workload(
        "random", np.zeros(3), np.ones(3), np.ones(3, np.int32), rng.uniform(0, 1, (3, n)),
        rng.uniform(0.06, 0.2, n), workloads.configs.background(n), 5.0 / 3.0)
    w.periodic[:] = periodic
    check(w, sets(phb, w), sample(w.n, min(w.n, 500), seed=2))


@pytest.mark.parametrize("ell", [8, 40])
def test_lists_longer_than_their_rows(ell):
    phb = need_gpu()
    w = workloads.shock_tube(5000, seed=9)
    check(w, sets(phb, w, ell_width=ell), sample(w.n, 500, seed=3))


def test_crowded_cells_and_lost_particles():
    """3,000 particles within a hundredth of a cell, and 2,500 whose positions
    are not numbers: the order inside the crowd's cell is by caller index, the
    lists of the others are those of the rest of the set."""
    phb = need_gpu()
    rng = np.random.default_rng(4)
    n = 9000
    w = workloads.Workload("crowd", np.zeros(3), np.ones(3), np.ones(3, np.int32), rng.uniform(0, 1, (3, n)),
                           rng.uniform(0.02, 0.03, n), workloads.configs.background(n), 5.0 / 3.0)
    crowd = rng.permutation(n)[:3000]
    w.pos[:, crowd] = 0.51 + 4e-4 * rng.uniform(-1, 1, (3, 3000))
    lost = np.setdiff1d(np.arange(n), crowd)[::2][:2500]
    pos = w.pos.copy()
    pos[0, lost] = np.nan
    plan = phb.Plan.for_workload(w, nbr_capacity=12_000_000)
    p, lam = torch.tensor(pos, device="cuda"), torch.tensor(w.lam, device="cuda")
    with pytest.raises(phb.PhbError):   # the non-finite positions are reported
        phb.build_neighbors(plan, p, lam)
    got = sets_of(*phb.export_neighbors(plan))
    keep = np.setdiff1d(np.arange(n), lost)
    off, idx = oracle.neighbors(oracle.box_of(w), w.pos[:, keep], w.lam[keep], np.arange(keep.size))
    for k in sample(keep.size, 300, seed=5):
        np.testing.assert_array_equal(got[keep[k]], keep[idx[off[k]:off[k + 1]]])
    assert all(got[i].size == 0 for i in lost[:50])
    pos_r, lam_r, U_r = p.clone(), lam.clone(), torch.tensor(w.U, device="cuda")
    perm = phb.reorder(plan, pos_r, lam_r, U_r).cpu().numpy()
    at = np.empty(n, np.int64)
    at[perm] = np.arange(n)
    assert np.array_equal(np.sort(perm), np.arange(n))
    # the crowd shares one cell: its storage order is by caller index
    assert (np.diff(at[np.sort(crowd)]) > 0).all()


@pytest.mark.parametrize("lengths,periodic", [((40.0, 1.0, 1.0), (1, 1, 1)), ((1.0, 1.0, 23.0), (0, 0, 0)),
                                              ((1.0, 34.5, 0.9), (0, 1, 0))])
def test_keys_of_the_grids_own_bricks(lengths, periodic):
    """Boxes whose Hilbert cube holds many more bricks than the grid, on both
    sides of the line from which keys are ranks of the grid's bricks: wrong
    ranks would merge or lose cells."""
    phb = need_gpu()
    rng = np.random.default_rng(11)
    n, L = 20_003, np.array(lengths)
    w = workloads.Workload("long", -0.3 * L, 0.7 * L, np.array(periodic, np.int32),
                           (rng.uniform(-0.3, 0.7, (n, 3)) * L).T.copy(), rng.uniform(0.06, 0.09, n),
                           workloads.configs.background(n), 5.0 / 3.0)
    plan = phb.Plan.for_workload(w)
    cube, bricks = 8 ** plan.c.hilbert_bits, int(np.prod(list(plan.c.nbrick)))
    assert plan.c.nkeys == 64 * (bricks if cube >= 2 ** 15 and 4 * bricks <= cube else cube)
    check(w, sets(phb, w), sample(n, 500, seed=6))
