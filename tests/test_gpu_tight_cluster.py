"""FP64 fits of neighbours that lie within 1e-7 lambda of the particle: entries
of the normal matrix (1e-47) that FP32 does not hold."""
import itertools

import numpy as np
import pytest

import workloads
from _gpu import need_gpu

pytestmark = pytest.mark.gpu

POWERS = [e for d in (1, 2, 3) for e in itertools.product(range(d, -1, -1), repeat=3) if sum(e) == d]


def derivs_by_qr(x, U, lam):
    """Gradients and Hessians (packed xx, xy, xz, yy, yz, zz) of particles that all
    list each other: weighted least squares of scaled columns, no normal equations."""
    n = x.shape[1]
    g, h = np.empty((8, 3, n)), np.empty((8, 6, n))
    for i in range(n):
        q = np.delete(x - x[:, i:i + 1], i, 1) / lam
        rw = 1.0 - (q * q).sum(0) / 2.3**2
        A = np.stack([rw * q[0]**a * q[1]**b * q[2]**c for a, b, c in POWERS], 1)
        s = 1.0 / np.linalg.norm(A, axis=0)
        rhs = (rw * np.delete(U - U[:, i:i + 1], i, 1)).T
        c = s[:, None] * np.linalg.lstsq(A * s, rhs, rcond=None)[0]
        g[:, :, i] = c[:3].T / lam
        h[:, :, i] = (c[3:9] * np.array([2, 1, 1, 2, 1, 2])[:, None]).T / lam**2
    return g, h


@pytest.mark.parametrize("others", [0, 6000])   # the warp form, the thread form
def test_corrected_step_of_a_tight_cluster(others):
    """21 particles for 19 coefficients: Jacobi-scaled condition estimates of 6e4
    and more, above the 1e4 from which the corrected step is taken; without it
    the worst error is 2e-11 (normal equations in numpy), with it 2e-14."""
    phb = need_gpu()
    x = 2e-9 * np.random.default_rng(0).uniform(0, 1, (21, 3)).T
    t = x / 2e-9
    rest = np.random.default_rng(1).uniform(0.2, 0.8, (3, others))
    n, lam = 21 + others, 0.05
    U = workloads.configs.background(n)
    for f in range(8):
        U[f, :21] += 0.1 * np.sin(3 * t[0] + (6 - 0.3 * f) * t[1] + 1.5 * t[2] + f)
    w = workloads.Workload("tight", np.zeros(3), np.ones(3), np.zeros(3, np.int32), np.concatenate([x, rest], 1),
                           np.full(n, lam), U, 5.0 / 3.0)
    plan = phb.Plan.for_workload(w, nbr_capacity=400 * n)
    p, l, u = phb.tensors_of(w)
    phb.build_neighbors(plan, p, l)
    g, h, st = phb.mls_derivs(plan, phb.Params(gamma=w.gamma, precision="fp64"), p, l, u)
    assert not st[:21].any()
    go, ho = derivs_by_qr(x, U[:, :21], lam)
    for a, o in ((g, go), (h, ho)):
        e = np.abs(a[:, :, :21].cpu().numpy() - o).max(axis=1) / np.abs(o).max(axis=1)
        assert e.max() < 1e-12, e.max()
