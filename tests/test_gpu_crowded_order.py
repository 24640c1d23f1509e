"""The order inside a cell on both sides of the line (members^2 = 256 n) from
which it comes from a sweep over all keys instead of each member's rank."""
import numpy as np
import pytest

import workloads
from _gpu import need_gpu, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,members", [(257, 256), (257, 257), (4000, 1011), (4000, 1012), (4000, 1013),
                                       (70_001, 4233), (70_001, 4234)])
@pytest.mark.parametrize("lost", [False, True])
def test_order_inside_a_crowded_cell(n, members, lost):
    """Members within one cell (few lists: a tiny lambda), or without a finite
    position, stand by caller index; each particle has one slot."""
    phb = need_gpu()
    rng = np.random.default_rng(members)
    pos = rng.uniform(0.0, 1.0, (3, n))
    crowd = np.sort(rng.permutation(n)[:members])
    pos[:, crowd] = 0.52 + 1e-4 * rng.uniform(-1, 1, (3, members))
    if lost:
        pos[2, crowd] = np.nan
    plan = phb.Plan((0, 0, 0), (1, 1, 1), (1, 1, 1), n, 1e-7, 1e-7, cell_frac=4e5)
    p = torch.tensor(pos, device="cuda")
    lam = torch.full((n,), 1e-7, dtype=torch.float64, device="cuda")
    U = torch.tensor(workloads.configs.background(n), device="cuda")
    phb.build_neighbors(plan, p, lam, check_capacity=False)
    perm = phb.reorder(plan, p, lam, U).cpu().numpy()
    assert np.array_equal(np.sort(perm), np.arange(n))
    at = np.empty(n, np.int64)
    at[perm] = np.arange(n)
    assert (np.diff(at[crowd]) > 0).all()
    if lost:
        assert np.array_equal(perm[n - members:], crowd)
