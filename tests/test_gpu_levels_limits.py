"""Time-step levels at the limits of FP64: an infinite dt_max (every level of it
is infinite: the deepest one) with steps up to 2^1020."""
import numpy as np
import pytest

import workloads
from _gpu import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dt_max,level", [(float("inf"), 20), (1e308, None)])
def test_infinite_dt_max(dt_max, level):
    phb = need_gpu()
    n, big, cfl, gamma = 5, 2.0**500, 0.25, 5.0 / 3.0
    U = workloads.configs.background(n)
    U[4:7] = 0.0
    U[7] = np.ldexp(1.0, -np.array([200, 900, 950, 1000, 1036]))
    pos = big * np.linspace(0.1, 0.9, 3 * n).reshape(3, n)
    w = workloads.Workload("far", np.zeros(3), np.full(3, 1e4 * big), np.zeros(3, np.int32), pos,
                           np.full(n, 1e-3 * big), U, gamma)
    plan = phb.Plan.for_workload(w)
    p, lam, u = phb.tensors_of(w)
    phb.build_neighbors(plan, p, lam, check_capacity=False)
    lv = phb.timestep_levels(plan, phb.Params(gamma=gamma), p, lam, u, cfl=cfl, dt_max=dt_max, max_level=20)
    dt = cfl * w.lam / np.sqrt(gamma * ((gamma - 1.0) * U[7]) / U[0])
    assert dt.max() > 2.0**994
    exp = [next(L for L in range(21) if L == 20 or dt_max / 2.0**L <= d) for d in dt]
    assert level is None or exp == [level] * n
    np.testing.assert_array_equal(lv.cpu().numpy(), exp)
