"""Where a workspace may start: any multiple of 16 bytes (its records, read 32
bytes at a time, are aligned inside it); anything else is refused on the host."""
import ctypes as C

import pytest

import workloads
from _gpu import need_gpu, torch


def test_other_addresses_are_refused_before_any_cuda_call():
    from paper_1110_0836_gb300 import _build, _lib
    _build.build()
    L = _lib.lib()
    p = _lib.Plan()
    for k in range(3):
        p.box.len[k], p.box.periodic[k] = 1.0, 1
    p.n, p.rf_factor, p.lambda_min, p.lambda_max, p.nbr_capacity = 4096, 2.3, 1 / 16, 1 / 16, 1 << 18
    assert L.phb_plan_init(C.byref(p)) == 0
    prm = _lib.Params()
    prm.gamma = 5.0 / 3.0
    arr = C.c_void_p(0x2000)
    for at in (0x1001, 0x1004, 0x1008, 0x100f):
        ws = C.c_void_p(at)
        assert L.phb_build_neighbors(C.byref(p), arr, arr, ws, p.ws_bytes, None, None) == _lib.PHB_ERR_INVALID_ARG
        assert L.phb_mhd_rhs(C.byref(p), C.byref(prm), arr, arr, arr, ws, p.ws_bytes, arr, None, None,
                             None) == _lib.PHB_ERR_INVALID_ARG
    # the records' region holds their shift; the address is read before the size
    off, nbytes = C.c_size_t(), C.c_size_t()
    assert L.phb_record_region(C.byref(p), C.byref(off), C.byref(nbytes)) == 0
    after = min(o for o in list(p.ws_off) if o > off.value)
    assert off.value + nbytes.value + 16 <= after
    assert L.phb_build_neighbors(C.byref(p), arr, arr, C.c_void_p(0x1010), 16, None, None) == _lib.PHB_ERR_WORKSPACE


@pytest.mark.gpu
@pytest.mark.parametrize("shift", [16, 48, 240])
def test_a_workspace_at_a_multiple_of_16_bytes(shift):
    """Staged tiles, the corrected step's two schedules and the unstaged path of
    an active subset read the records: the same results, bit for bit."""
    phb = need_gpu()
    w = workloads.shock_tube(4001, seed=8)
    pos, lam, U = phb.tensors_of(w)
    idx = torch.arange(0, w.n, 3, dtype=torch.int32, device="cuda")
    out = []
    for s in (0, shift):
        plan = phb.Plan.for_workload(w)
        whole = torch.empty(plan.ws.numel() + s, dtype=torch.uint8, device="cuda")
        plan.ws = whole[s:]
        assert plan.ws.data_ptr() % 256 == s
        phb.build_neighbors(plan, pos, lam)
        for sched in ("queue", "tile"):
            prm = phb.Params(gamma=w.gamma, refine="on", refine_schedule=sched)
            out.append(phb.mhd_rhs(plan, prm, pos, lam, U)[0].clone())
            out.append(phb.mhd_rhs_active(plan, prm, pos, lam, U, idx)[:, ::3].clone())
        p, u = pos.clone(), U.clone()
        phb.pc_step(plan, phb.Params(gamma=w.gamma), p, lam, u, 1e-6)
        out += [p, u]
    assert len(out) == 12 and all(torch.equal(a, b) for a, b in zip(out[:6], out[6:]))
