"""Size of the adjoint's part of the workspace: below the stored record it
avoids but for small sets, bounded for those, and without a jump."""
import ctypes as C

import pytest


def part(n, capacity):
    from paper_1110_0836_gb300 import _build, _lib
    _build.build()
    p = _lib.Plan()
    for k in range(3):
        p.box.len[k], p.box.periodic[k] = 1.0, 1
    lam = min(n ** (-1 / 3), 0.2)
    p.n, p.rf_factor, p.lambda_min, p.lambda_max = n, 2.3, lam, lam
    p.nbr_capacity = capacity if capacity else 72 * n + 1024
    assert _lib.lib().phb_plan_init(C.byref(p)) == 0
    b, e = _lib.workspace_part(p, _lib.PART_ADJOINT)
    return e - b, _lib.lib().phb_adjoint_record_bytes(C.byref(p))


@pytest.mark.parametrize("capacity", [None, 1 << 30])
@pytest.mark.parametrize("n", [36_000, 60_000, 100_003, (1 << 17) - 1, 1 << 17, (1 << 17) + 1, 1 << 18, 8_000_000])
def test_less_than_the_record(n, capacity):
    size, record = part(n, capacity)
    assert size < record


@pytest.mark.parametrize("n", [1, 2, 100, 1000, 4096, 14_000, 19_456, 30_000, 37_449, 37_450])
def test_small_sets_are_bounded(n):
    size, record = part(n, None)
    assert size < max(record, (84 << 20) + 120 * n + 4096)
    for more in (n + 1, n + 2):
        assert abs(part(more, None)[0] - size) < 16_000   # a particle's list and its own words
    assert part(n, 1 << 30)[0] < (84 << 20) + 120 * n + 4096 + (84 * 28 * n if n > 37_449 else 0)
