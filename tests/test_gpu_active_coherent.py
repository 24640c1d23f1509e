"""Active subsets that are coherent in space (runs of the storage order), on both
sides of half of the particles."""
import pytest

import workloads
from _gpu import need_gpu, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("share", [0.02, 0.4, 0.5, 0.51])
@pytest.mark.parametrize("which", ["lattice", "tube"])
def test_runs_of_the_storage_order(which, share):
    """Within the FP32-mixed bound (two evaluations of 1e-5 each) of the whole
    set's evaluation; above half its tiles, bit for bit; other columns left alone."""
    phb = need_gpu()
    w = workloads.random_modes(17, seed=92, amp=0.05) if which == "lattice" else workloads.shock_tube(9001, seed=92)
    n = w.n
    plan = phb.Plan.for_workload(w)
    pos, lam, U = phb.tensors_of(w)
    phb.build_neighbors(plan, pos, lam)
    phb.reorder(plan, pos, lam, U)
    phb.build_neighbors(plan, pos, lam)
    prm = phb.Params(gamma=w.gamma)
    full, _ = phb.mhd_rhs(plan, prm, pos, lam, U)
    k = int(share * n)
    a = n // 5   # neither end on a tile
    act = torch.arange(a, a + k, dtype=torch.int32, device="cuda")
    out = phb.mhd_rhs_active(plan, prm, pos, lam, U, act, out=torch.full((8, n), 7.5, dtype=torch.float64, device="cuda"))
    got, exp = out[:, a:a + k], full[:, a:a + k]
    assert bool((out[:, :a] == 7.5).all()) and bool((out[:, a + k:] == 7.5).all())
    if 2 * k > n:
        assert torch.equal(got, exp) or which == "tube"   # a tile's corrected step is decided by its active fits
    scale = full.abs().amax(dim=1, keepdim=True)
    scale = torch.maximum(scale, 1e-2 * scale.max())   # the tests' floor: fields that vanish
    assert float(((got - exp).abs() / scale).max()) < 2e-5
