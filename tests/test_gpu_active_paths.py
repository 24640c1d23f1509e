"""Active subsets on either side of half of the particles, where the FP32-mixed
fit changes from listed slots to whole tiles."""
import numpy as np
import pytest

import workloads
from _gpu import need_gpu, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile", [64, 128])
@pytest.mark.parametrize("share", ["none", "half", "half + 1", "run", "all"])
def test_active_shares(share, tile):
    """Up to half: listed slots, within the FP32-mixed bound of the full
    evaluation.  More than half (at random, or a run that leaves whole tiles
    without active particles): the full evaluation's tiles, bit for bit.  Other
    columns are left alone."""
    phb = need_gpu()
    w = workloads.random_modes(15, seed=91, amp=0.05)   # 3,375: a partial last tile
    n = w.n
    plan = phb.Plan.for_workload(w, tile=tile, cell_frac=0.5)
    pos, lam, U = phb.tensors_of(w)
    phb.build_neighbors(plan, pos, lam)
    prm = phb.Params(gamma=w.gamma)
    full, _ = phb.mhd_rhs(plan, prm, pos, lam, U)
    rng = np.random.default_rng(3)
    idx = {"none": np.zeros(0), "half": rng.permutation(n)[:n // 2], "half + 1": rng.permutation(n)[:n // 2 + 1],
           "run": np.arange(n - (2 * n) // 3, n), "all": np.arange(n)}[share].astype(np.int32)
    mark = torch.zeros(n, dtype=torch.bool, device="cuda")
    act = torch.tensor(idx, device="cuda")
    mark[act.long()] = True
    out = torch.full((8, n), 7.5, dtype=torch.float64, device="cuda")
    phb.mhd_rhs_active(plan, prm, pos, lam, U, act, out=out)
    assert bool((out[:, ~mark] == 7.5).all())
    if 2 * idx.size > n:
        assert torch.equal(out[:, mark], full[:, mark])
    elif idx.size:
        scale = full.abs().amax(dim=1, keepdim=True)
        assert float(((out - full)[:, mark].abs() / scale).max()) < 2e-5   # two evaluations of 1e-5 each
