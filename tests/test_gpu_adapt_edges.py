"""Adaptivity scan and time-step levels where their kernels change path: few
particles, lists beyond two rounds of a warp, void factors whose test-point
limits coincide with grid radii (each particle's own rounding decides), and
levels at exact powers of two, against the exact oracle."""
import numpy as np
import pytest

import oracle
import workloads
from _gpu import need_gpu, torch

pytestmark = pytest.mark.gpu


def random_set(n, lam, seed):
    rng = np.random.default_rng(seed)
    U = workloads.configs.background(n)
    return workloads.Workload("random", np.zeros(3), np.ones(3), np.ones(3, np.int32),
                              rng.uniform(0.0, 1.0, (3, n)), np.asarray(lam(rng, n)), U, 5.0 / 3.0)


@pytest.mark.parametrize("n,lam0", [(1, 0.1), (33, 0.15), (2000, 0.08), (900, 0.16)])
@pytest.mark.parametrize("vf", [1.0, 1.15, 0.575, 0.3])
def test_scan_exact(n, lam0, vf):
    """2.3 lambda / 4 = 0.575 lambda: for vf = 1.15 the points with |k| = 2 lie on
    both limits, for 0.575 those with |k| = 1 and 3; 0.3 reaches |k|^2 = 12."""
    phb = need_gpu()
    w = random_set(n, lambda rng, n: lam0 * rng.uniform(0.8, 1.25, n), seed=n)
    plan = phb.Plan.for_workload(w)
    pos, lam, _ = phb.tensors_of(w)
    phb.build_neighbors(plan, pos, lam)
    got = [o.cpu().numpy() for o in phb.adapt_scan(plan, pos, lam, void_factor=vf, clump_factor=0.25)]
    box = oracle.box_of(w)
    exp = oracle.adapt_scan(box, w.pos, w.lam, oracle.neighbors(box, w.pos, w.lam), None, void_factor=vf,
                            clump_factor=0.25)
    for a, b in zip(got, exp):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("max_level", [0, 3, 30])
def test_levels_at_powers_of_two(max_level):
    """Steps that are dt_max / 2^L exactly, one bit below and one above, and far
    outside the range of levels."""
    phb = need_gpu()
    n = 96
    w = random_set(n, lambda rng, n: np.full(n, 1e-3), seed=5)   # no neighbours: unlimited levels
    # gamma P + B^2 = c^2 rho with P = (gamma - 1) sigma, B = 0: dt = cfl lambda / c
    c = np.ldexp(1.0, np.arange(n) // 3 - 40) * (1.0 + np.array([-2.0**-52, 0.0, 2.0**-52])[np.arange(n) % 3])
    w.U[4:7] = 0.0
    w.U[7] = c * c / (w.gamma * (w.gamma - 1.0))
    plan = phb.Plan.for_workload(w)
    pos, lam, U = phb.tensors_of(w)
    phb.build_neighbors(plan, pos, lam)
    dt_max = 0.25 * 1e-3 * 2.0**20
    lv = phb.timestep_levels(plan, phb.Params(gamma=w.gamma), pos, lam, U, cfl=0.25, dt_max=dt_max,
                             max_level=max_level)
    nb = oracle.neighbors(oracle.box_of(w), w.pos, w.lam)
    exp = oracle.timestep_levels(w.lam, w.U, nb, gamma=w.gamma, cfl=0.25, dt_max=dt_max, max_level=max_level)
    np.testing.assert_array_equal(lv.cpu().numpy(), exp)
    assert max_level < 30 or len(np.unique(exp)) > 8
