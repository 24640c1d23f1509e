"""Adaptivity with a lambda that is not a positive number: such a particle has
no test points (each of the definition's comparisons is false), so it marks no
void and creates nothing; the other particles are not touched by it."""
import numpy as np
import pytest

import workloads
from _gpu import need_gpu, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("built", [False, True])
@pytest.mark.parametrize("vf", [1.0, 0.3])
def test_scan_and_apply(vf, built):
    """The lambda lost before the build (no list), or after it (a list)."""
    phb = need_gpu()
    rng = np.random.default_rng(6)
    n = 3000
    w = workloads.Workload("holes", np.zeros(3), np.ones(3), np.ones(3, np.int32), rng.uniform(0, 1, (3, n)),
                           0.07 * rng.uniform(0.9, 1.1, n), workloads.configs.background(n), 5.0 / 3.0)
    plan = phb.Plan.for_workload(w)
    pos, lam, U = phb.tensors_of(w)
    phb.build_neighbors(plan, pos, lam)
    ref = [o.clone() for o in phb.adapt_scan(plan, pos, lam, void_factor=vf)]
    assert int((ref[0] > 0).sum()) > n // 10
    at = torch.tensor(rng.permutation(n)[:12], device="cuda")
    lam[at] = torch.tensor([np.nan, np.inf, 0.0, -np.inf] * 3, dtype=torch.float64, device="cuda")
    if built:
        with pytest.raises(phb.PhbError):
            phb.build_neighbors(plan, pos, lam)
    scan = phb.adapt_scan(plan, pos, lam, void_factor=vf)
    vc, best, cand, clump = scan
    other = torch.ones(n, dtype=torch.bool, device="cuda")
    other[at] = False
    for a, b in zip(scan, ref):
        assert torch.equal(a[..., other], b[..., other])
    assert not bool(vc[at].any()) and bool((best[at] == -1).all()) and not bool(cand[:, at].any())
    g, h, _ = phb.mls_derivs(plan, phb.Params(gamma=w.gamma, precision="fp64"), pos, lam, U)
    p2, l2, _, org = phb.adapt_apply(plan, pos, lam, U, scan, g, h, void_factor=vf)
    made = org[org >= n] - n
    assert made.numel() > 0 and not bool(torch.isin(made, at).any())
    assert bool(torch.isfinite(p2).all()) and int((~torch.isfinite(l2)).sum()) <= 9
