"""The FP64 fit's two forms (a thread per particle, a warp per particle) and
the adjoint's reverse lists at the sizes where their paths change."""
import numpy as np
import pytest

import oracle
import workloads
from _gpu import need_gpu, rhs_err, rhs_term_scales, sample, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("which", [8, 17, 28, "tube", "open"])
def test_thread_and_warp_forms_agree(which):
    """The right-hand side of all particles (512: warp form; 4,913: thread form;
    21,952: a full pass of the thread form and a remainder for the warp form;
    varying lists; one-sided and singular fits) equals, bit for bit, that of
    300 listed ones (warp form), and both meet 1e-12 against the oracle."""
    phb = need_gpu()
    w = workloads.shock_tube(20_001, seed=61) if which == "tube" else \
        workloads.random_modes(17 if which == "open" else which, seed=61, amp=0.05)
    if which == "open":
        w.periodic[:] = 0
    plan = phb.Plan.for_workload(w)
    pos, lam, U = phb.tensors_of(w)
    phb.build_neighbors(plan, pos, lam)
    prm = phb.Params(gamma=w.gamma, precision="fp64")
    st = torch.empty(w.n, dtype=torch.int32, device="cuda")
    out, _ = phb.mhd_rhs(plan, prm, pos, lam, U, fit_status=st)
    q = sample(w.n, 300, seed=5)
    sa = torch.zeros_like(st)
    part = phb.mhd_rhs_active(plan, prm, pos, lam, U, torch.tensor(q, dtype=torch.int32, device="cuda"),
                              fit_status=sa)
    assert torch.equal(out[:, q], part[:, q]) and torch.equal(st[q], sa[q])
    box = oracle.box_of(w)
    nb = oracle.neighbors(box, w.pos, w.lam, q)
    exp, sto = oracle.mhd_rhs(box, w.pos, w.lam, w.U, nb, q, gamma=w.gamma)
    assert np.array_equal(sto, st[q].cpu().numpy())
    g, h, _ = oracle.mls_derivs(box, w.pos, w.lam, w.U, nb, q, gamma=w.gamma)
    # one-sided fits at open faces: the bound of the other open-box test
    tol = 1e-8 if which == "open" else 1e-12
    e = rhs_err(out[:, q].cpu().numpy(), exp, rhs_term_scales(w.U[:, q], g, h, w.gamma))
    assert e.max() < tol, e


@pytest.mark.parametrize("capacity", [None, 20_000_000])
def test_adjoint_long_reverse_lists(capacity):
    """Particles named by more lists than a warp keeps in registers (128), and a
    capacity whose entries go through the term buffer in several chunks (the
    later ones empty): <gbar, J v> of the oracle equals <J^T gbar, v>."""
    phb = need_gpu()
    rng = np.random.default_rng(71)
    n = 700
    pos = rng.uniform(0.0, 1.0, (3, n))
    U = workloads.configs.background(n)
    x = 2 * np.pi * pos
    for f in range(8):
        U[f] += 0.05 * np.sin(x[f % 3] + f) * np.cos(x[(f + 1) % 3])
    w = workloads.Workload("dense", np.zeros(3), np.ones(3), np.ones(3, np.int32), pos,
                           np.full(n, 0.18), U, 5.0 / 3.0)
    plan = phb.Plan.for_workload(w, nbr_capacity=capacity)
    p, lam, u = phb.tensors_of(w)
    phb.build_neighbors(plan, p, lam)
    off, idx = phb.export_neighbors(plan)
    assert torch.bincount(idx.long()).max() > 128
    prm = phb.Params(gamma=w.gamma, precision="fp64")
    gbar = rng.standard_normal((8, n))
    Ub, xb = phb.rhs_adjoint(plan, prm, p, lam, u, torch.tensor(gbar, device="cuda"))
    vpos, vU = rng.standard_normal((3, n)) * w.lam, rng.standard_normal((8, n))
    box = oracle.box_of(w)
    _, jv = oracle.rhs_jvp(box, w.pos, w.lam, w.U, vpos, vU, oracle.neighbors(box, w.pos, w.lam),
                           gamma=w.gamma)
    lhs = float((gbar * jv).sum())
    rhs = float((Ub.cpu().numpy() * vU).sum() + (xb.cpu().numpy() * vpos).sum())
    assert abs(lhs - rhs) <= 1e-10 * max(abs(lhs), 1.0), (lhs, rhs)
