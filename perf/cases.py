"""Timed cases: what a simulation or an inference program asks of this package.

The particle sets are those of the package's own workloads (jittered lattice
with random Fourier modes, Brio-Wu-like shock tube, Kelvin-Helmholtz shear
layer), drawn on the GPU.  `exact` restates the method (neighbour sets, cubic
interpolating MLS fit, Lagrangian MHD time derivatives, Heun steps) in plain
64-bit torch.
"""
import math

import torch

import paper_1110_0836_gb300 as phb

DEV = "cuda"
RF = 2.3          # r_f / lambda
NBR = 4.0 / 3.0 * math.pi * RF ** 3   # neighbours per particle at density 1 / lambda^3
VOID, CLUMP = 1.0, 0.25               # adaptivity thresholds (the defaults of adapt_scan)
CFL = 0.002       # steps advance in place: short ones keep a state the same kind of state over many passes
LAWS = dict(c_zeta_l=0.1, c_zeta_a=1.0, c_eta=0.1)


def listed():
    return [
        # a convergence test's inner loop: 4,096 particles, captured steps, launch latency
        dict(name="step_16", kind="step", set="lattice", side=16),
        # the same small scale without a graph: a shock tube with fixed-value ends and viscosity laws
        dict(name="step_tube_open", kind="eager", set="tube", n=10_007, open=True),
        # the benchmark's lattice step, captured
        dict(name="step_64", kind="step", set="lattice", side=64),
        # the benchmark's end-to-end step: state in pinned host memory
        dict(name="host_64", kind="host", set="lattice", side=64),
        # varying resolution, every fit refined
        dict(name="step_tube", kind="step", set="tube", n=1 << 20),
        # the largest set: a production run's step
        dict(name="step_layer", kind="eager", set="layer", n=8_000_000),
        # individual time steps: levels, then one synchronised step of four substeps
        dict(name="block_layer", kind="block", set="layer", n=200_000),
        # right-hand side in double precision (validation runs, small amplitudes)
        dict(name="rhs64_64", kind="rhs64", set="lattice", side=64),
        # gradients and Hessians of all fields in double precision (analysis, refinement states)
        dict(name="derivs64_tube", kind="derivs64", set="tube", n=60_000),
        # inference: forward and reverse mode with recomputed factorisations
        dict(name="grad_64", kind="grad", set="lattice", side=64, stored=False),
        # the same from stored factorisations, on a set of varying resolution
        dict(name="grad_stored_tube", kind="grad", set="tube", n=100_003, stored=True),
        # what a run checks every few steps: voids, clumps and time-step levels
        dict(name="scan_tube", kind="scan", set="tube", n=400_000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "eager", "eager", "host", "block", "rhs64", "derivs64", "grad", "scan"])
    # sharply refined sets leave a few fits that are ill-conditioned in themselves: double precision and
    # gradients are asked of the other two
    which = rng.choice(["lattice", "tube"] if kind in ("rhs64", "derivs64", "grad") else ["lattice", "tube", "layer"])
    lo, hi = {"step": (4e3, 2e6), "eager": (4e3, 4e6), "host": (4e3, 1e6), "block": (8e3, 3e5),
              "rhs64": (4e3, 2.5e5), "derivs64": (4e3, 2e5), "grad": (4e3, 1.5e5), "scan": (4e3, 1e6)}[kind]
    n = _log_int(rng, lo, hi)
    case = dict(kind=kind, set=which)
    if which == "lattice":
        case["side"] = round(n ** (1.0 / 3.0))
    else:
        case["n"] = n
    if kind == "eager":
        case["open"] = which == "tube" and rng.random() < 0.5
    if kind == "grad":
        case["stored"] = rng.random() < 0.5
    return case


def _count(case):
    return case["side"] ** 3 if case["set"] == "lattice" else case["n"]


def work(case):
    n, kind = _count(case), case["kind"]
    # per particle: 80 moments and the fields' right-hand sides over the neighbours, offsets and
    # monomials, factorisation and solves
    rhs = NBR * (2 * (80 + 7 * 19) + 60) + 2300 + 7 * 600
    derivs = NBR * (2 * (80 + 8 * 19) + 60) + 2300 + 8 * 600
    back = NBR * (2 * (2 * 7 * 19 + 200) + 60) + 7 * 1400 + 2 * 7 * 361
    # per particle: x, lambda, U in (12 words), and what comes out
    flops, words = {
        "step": (2 * rhs, 12 + 11), "eager": (2 * rhs, 12 + 11), "host": (2 * rhs, 12 + 11),
        # one evaluation at the start, then at least two for the particles of the shortest steps
        "block": (3 * rhs, 12 + 11 + 0.5), "rhs64": (rhs, 12 + 8), "derivs64": (derivs, 12 + 72.5),
        "grad": (rhs + back, 12 + 8 + 8 + 11), "scan": (NBR * 57 * 8, 12 + 5)}[kind]
    return {"bytes": 8.0 * words * n, "flops": float(flops * n)}


# ---------------------------------------------------------------- particle sets

def _uniform(gen, shape, lo=0.0, hi=1.0):
    return lo + (hi - lo) * torch.rand(shape, generator=gen, device=DEV, dtype=torch.float64)


def _background(n, gamma):
    U = torch.zeros((8, n), dtype=torch.float64, device=DEV)
    U[0], U[4], U[5], U[6], U[7] = 1.0, 1.0, math.sqrt(2.0), 0.5, 1.0 / (gamma - 1.0)
    return U


def _lattice(side, gen):
    """Jittered lattice in the periodic unit box, eight random Fourier modes on a uniform state."""
    gamma, h, n = 5.0 / 3.0, 1.0 / side, side ** 3
    k = torch.arange(side, dtype=torch.float64, device=DEV)
    grid = torch.stack(torch.meshgrid(k, k, k, indexing="ij")).reshape(3, n)
    pos = (grid + 0.5) * h + _uniform(gen, (3, n), -0.1 * h, 0.1 * h)
    U = _background(n, gamma)
    kv = torch.randint(-4, 5, (8, 3), generator=gen, device=DEV).double()
    kv[:, 0] += (kv.abs().sum(1) == 0).double()
    a, phi = _uniform(gen, (8, 8), -1e-2, 1e-2), _uniform(gen, (8,), 0.0, 2.0 * math.pi)
    for m in range(8):
        wave = torch.sin(2.0 * math.pi * (kv[m, 0] * pos[0] + kv[m, 1] * pos[1] + kv[m, 2] * pos[2]) + phi[m])
        U += a[m][:, None] * wave
    return ((0.0, 0.0, 0.0), (1.0, 1.0, 1.0), (1, 1, 1)), pos, torch.full((n,), h, dtype=torch.float64, device=DEV), U, gamma


def _interp(x, xp, fp):
    i = torch.searchsorted(xp, x).clamp(1, xp.numel() - 1)
    return fp[i - 1] + (fp[i] - fp[i - 1]) * (x - xp[i - 1]) / (xp[i] - xp[i - 1])


def _tube(n, gen, open_ends):
    """Brio-Wu-like tube, 8 x 1 x 1, two mirrored interfaces, lambda = lambda_L rho^(-1/3), density-sampled."""
    gamma, lam_l = 2.0, (4.5 / n) ** (1.0 / 3.0)
    w = 2.0 * lam_l

    def s_of(x):
        return 0.5 * (torch.tanh((x - 2.0) / w) - torch.tanh((x - 6.0) / w))

    grid = torch.linspace(0.0, 8.0, (1 << 18) + 1, dtype=torch.float64)
    dens = 1.0 - 0.875 * s_of(grid)
    cdf = torch.cat([dens.new_zeros(1), torch.cumsum(0.5 * (dens[1:] + dens[:-1]), 0)])  # on the CPU: the same sums each time
    x = _interp(_uniform(gen, (n,)), (cdf / cdf[-1]).to(DEV), grid.to(DEV))
    pos = torch.stack([x, _uniform(gen, (n,)), _uniform(gen, (n,))])
    s = s_of(x)
    U = torch.zeros((8, n), dtype=torch.float64, device=DEV)
    U[0], U[4], U[5], U[7] = 1.0 - 0.875 * s, 0.75, 1.0 - 2.0 * s, (1.0 - 0.9 * s) / (gamma - 1.0)
    return ((0.0, 0.0, 0.0), (8.0, 1.0, 1.0), (0 if open_ends else 1, 1, 1)), pos, lam_l * U[0] ** (-1.0 / 3.0), U, gamma


def _layer(n, gen):
    """Double shear layer in the periodic unit box, lambda halved within 0.1 of the layers, density-sampled."""
    gamma, lam0, w = 5.0 / 3.0, (3.8 / n) ** (1.0 / 3.0), 0.05
    yb = torch.tensor([0.0, 0.15, 0.35, 0.65, 0.85, 1.0], dtype=torch.float64, device=DEV)
    db = torch.tensor([1.0, 8.0, 1.0, 8.0, 1.0], dtype=torch.float64, device=DEV)
    cum = torch.cat([db.new_zeros(1), torch.cumsum(db * (yb[1:] - yb[:-1]), 0)])
    y = _interp(_uniform(gen, (n,)), cum / cum[-1], yb)
    pos = torch.stack([_uniform(gen, (n,)), y, _uniform(gen, (n,))])
    band = 0.5 * (torch.tanh((y - 0.25) / w) - torch.tanh((y - 0.75) / w))
    dy = torch.minimum((y - 0.25).abs(), (y - 0.75).abs())
    U = torch.zeros((8, n), dtype=torch.float64, device=DEV)
    U[0], U[1], U[4], U[7] = 1.0 + band, band - 0.5, 0.1, 2.5 / (gamma - 1.0)
    U[2] = 1e-2 * _uniform(gen, (n,), -1.0, 1.0) * torch.exp(-(dy / w) ** 2)
    lam = lam0 * torch.where(dy < 0.1, 0.5, 1.0).double()
    return ((0.0, 0.0, 0.0), (1.0, 1.0, 1.0), (1, 1, 1)), pos, lam, U, gamma


def _curve_order(box, pos, lam):
    """Particles along a Morton curve over cells of about one radius, as a tree code keeps them."""
    key = torch.zeros(pos.shape[1], dtype=torch.int64, device=DEV)
    for a in range(3):
        c = ((pos[a] - box[0][a]) / (RF * float(lam.min()))).long().clamp(0, 1023)
        for b in range(10):
            key |= ((c >> b) & 1) << (3 * b + a)
    return torch.sort(key, stable=True).indices


def _inputs(case, seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed) * 1000003 + 17)
    if case["set"] == "lattice":
        box, pos, lam, U, gamma = _lattice(case["side"], gen)
    elif case["set"] == "tube":
        box, pos, lam, U, gamma = _tube(case["n"], gen, case.get("open", False))
    else:
        box, pos, lam, U, gamma = _layer(case["n"], gen)
    order = _curve_order(box, pos, lam)
    pos, lam, U = pos[:, order].contiguous(), lam[order].contiguous(), U[:, order].contiguous()
    fast = ((gamma * (gamma - 1.0) * U[7] + (U[4:7] ** 2).sum(0)) / U[0]).sqrt()
    dt = CFL * float((lam / (fast + U[1:4].norm(dim=0))).min())
    vmax = float(U[1:4].norm(dim=0).max())
    skin = max(4.0 * dt * vmax, 0.02 * RF * float(lam.min()))
    frozen = None
    if case.get("open", False):  # fixed-value ends, a radius and a half wide
        frozen = (pos[0] < 1.5 * RF * lam) | (pos[0] > 8.0 - 1.5 * RF * lam)
    gbar = _uniform(gen, U.shape, -1.0, 1.0) if case["kind"] == "grad" else None
    return box, pos, lam, U, gamma, dt, skin, frozen, gbar


# ---------------------------------------------------------------- the calls

class _State:
    pass


def prepare(case, seed):
    kind = case["kind"]
    box, pos, lam, U, gamma, dt, skin, frozen, gbar = _inputs(case, seed)
    s = _State()
    s.kind, s.dt = kind, dt
    step = kind in ("step", "eager", "host")
    s.plan = phb.Plan(*box, pos.shape[1], float(lam.min()), float(lam.max()), skin=skin if step else 0.0)
    fp64 = kind in ("rhs64", "derivs64", "grad")
    s.params = phb.Params(gamma=gamma, precision="fp64" if fp64 else "fp32_mixed", frozen=frozen,
                          **(LAWS if frozen is not None else {}))
    s.pos, s.lam, s.U, s.gbar = pos, lam, U, gbar
    phb.build_neighbors(s.plan, pos, lam)  # sizes the plan's lists
    if kind in ("host", "eager") and frozen is None:
        phb.reorder(s.plan, pos, lam, U)   # the library's own storage order, once
    if kind == "step":
        s.graph = phb.StepGraph(s.plan, s.params, pos, lam, U, dt)
    elif kind == "host":
        host = [t.cpu().pin_memory() for t in (pos, lam, U)]
        s.out = [torch.empty_like(host[0]).pin_memory(), torch.empty_like(host[2]).pin_memory()]
        s.graph = phb.HostStepGraph(s.plan, s.params, *host, dt, *s.out)
    elif kind == "block":
        s.dt_max = _dt_max(lam, U, gamma)
        s.levels = torch.empty(pos.shape[1], dtype=torch.int32, device=DEV)
    elif kind == "grad":
        s.stored = case["stored"]
        s.pos.requires_grad_(True)
        s.U.requires_grad_(True)
    return s


def _dt_max(lam, U, gamma):
    """The step of the coarsest particles (level 0)."""
    fast = ((gamma * (gamma - 1.0) * U[7] + (U[4:7] ** 2).sum(0)) / U[0]).sqrt()
    return CFL * float((lam / fast).max())


def run(s):
    if s.kind == "step":
        s.graph.replay()
        return s.pos, s.U
    if s.kind == "eager":
        phb.pc_step(s.plan, s.params, s.pos, s.lam, s.U, s.dt)
        return s.pos, s.U
    if s.kind == "host":
        s.graph.replay()
        torch.cuda.synchronize()  # the outputs are in host memory
        return s.out
    phb.build_neighbors(s.plan, s.pos, s.lam, check_capacity=False)
    if s.kind == "block":
        phb.timestep_levels(s.plan, s.params, s.pos, s.lam, s.U, CFL, s.dt_max, 2, out=s.levels)
        phb.block_step(s.plan, s.params, s.pos, s.lam, s.U, s.levels, s.dt_max, 2)
        return s.pos, s.U, s.levels
    if s.kind == "rhs64":
        return phb.mhd_rhs(s.plan, s.params, s.pos, s.lam, s.U)[0]
    if s.kind == "derivs64":
        return phb.mls_derivs(s.plan, s.params, s.pos, s.lam, s.U)
    if s.kind == "grad":
        out = phb.rhs_autograd(s.pos, s.U, s.lam, s.plan, s.params, s.stored)
        return (out.detach(), *torch.autograd.grad(out, (s.pos, s.U), s.gbar))
    levels = phb.timestep_levels(s.plan, s.params, s.pos, s.lam, s.U, CFL, 0.01, 20)
    return (*phb.adapt_scan(s.plan, s.pos, s.lam, VOID, CLUMP), levels)


# ---------------------------------------------------------------- the same in plain 64-bit torch

MONO = [(a, b, d - a - b) for d in (1, 2, 3) for a in range(d, -1, -1) for b in range(d - a, -1, -1)]
LIN = [MONO.index(e) for e in ((1, 0, 0), (0, 1, 0), (0, 0, 1))]
QUAD = [MONO.index(e) for e in ((2, 0, 0), (1, 1, 0), (1, 0, 1), (0, 2, 0), (0, 1, 1), (0, 0, 2))]
HESS = [[0, 1, 2], [1, 3, 4], [2, 4, 5]]


def _offset(box, d):
    """Minimum image of offsets d [3, ...] on the periodic axes."""
    return torch.stack([d[a] - box[1][a] * torch.round(d[a] / box[1][a]) if box[2][a] else d[a] for a in range(3)])


def _square(d):
    return (d[0] * d[0] + d[1] * d[1]) + d[2] * d[2]


def _lists(box, pos, lam):
    """Neighbour sets {j != i: |x_j - x_i| < r_f,i} as (starts [n + 1], members)."""
    n, r = pos.shape[1], RF * lam
    nc = [max(1, int(box[1][a] // float(r.max()))) for a in range(3)]
    c = []
    for a in range(3):
        k = torch.floor((pos[a] - box[0][a]) / box[1][a] * nc[a]).long()
        c.append(k % nc[a] if box[2][a] else k.clamp(0, nc[a] - 1))
    cell = (c[0] * nc[1] + c[1]) * nc[2] + c[2]
    order = torch.argsort(cell)
    counts = torch.bincount(cell, minlength=nc[0] * nc[1] * nc[2])
    start, most = torch.cumsum(counts, 0) - counts, int(counts.max())
    table = torch.full((counts.numel(), most), -1, dtype=torch.int64, device=pos.device)
    table[cell[order], torch.arange(n, device=pos.device) - start[cell[order]]] = order
    steps = [(-1, 0, 1) if nc[a] >= 3 or not box[2][a] else range(nc[a]) for a in range(3)]
    size = max(1, (1 << 25) // (27 * most))
    got, lens = [], []
    for i0 in range(0, n, size):
        i = torch.arange(i0, min(i0 + size, n), device=pos.device)
        cand = []
        for sx in steps[0]:
            for sy in steps[1]:
                for sz in steps[2]:
                    k, ok = [], torch.ones_like(i, dtype=torch.bool)
                    for a, st in enumerate((sx, sy, sz)):
                        ka = c[a][i] + st
                        if box[2][a]:
                            ka = ka % nc[a]
                        else:
                            ok &= (ka >= 0) & (ka < nc[a])
                            ka = ka.clamp(0, nc[a] - 1)
                        k.append(ka)
                    t = table[(k[0] * nc[1] + k[1]) * nc[2] + k[2]]
                    cand.append(torch.where(ok[:, None], t, -1))
        cand = torch.cat(cand, 1)
        d2 = _square(_offset(box, pos[:, cand.clamp(min=0)] - pos[:, i, None]))
        hit = (cand >= 0) & (cand != i[:, None]) & (d2 < (r * r)[i, None])
        got.append(cand[hit])
        lens.append(hit.sum(1))
    lens = torch.cat(lens)
    return torch.cat([lens.new_zeros(1), torch.cumsum(lens, 0)]), torch.cat(got)


def _padded(lists, i):
    """(members [B, K], present [B, K]) of the sets of particles i (consecutive)."""
    off, mem = lists
    b, ln = off[i], off[i + 1] - off[i]
    k = torch.arange(max(1, int(ln.max())), device=off.device)
    there = k[None] < ln[:, None]
    return mem[torch.where(there, b[:, None] + k[None], 0)] if mem.numel() else torch.zeros_like(there, dtype=torch.int64), there


def _fit(box, pos, lam, U, lists, i, refine):
    """Gradients [8, 3, B] and Hessians [8, 6, B] of all fields at particles i."""
    j, there = _padded(lists, i)
    d = _offset(box, pos[:, j] - pos[:, i, None])
    s2 = _square(d) / ((RF * lam[i]) ** 2)[:, None]
    inside = there & (s2 < 1.0)
    w = torch.where(inside, (1.0 - s2) ** 2, 0.0)
    q = torch.where(inside, d / lam[i][:, None], 0.0)
    one = torch.ones_like(q[0])
    pw = [[one, q[a], q[a] * q[a], q[a] * q[a] * q[a]] for a in range(3)]
    P = torch.stack([pw[0][e[0]] * pw[1][e[1]] * pw[2][e[2]] for e in MONO], -1)
    du = (U[:, j] - U[:, i, None]).permute(1, 2, 0)
    WP = w[..., None] * P
    A = P.transpose(1, 2) @ WP
    ok = inside.sum(1) >= len(MONO)
    A = torch.where(ok[:, None, None], A, torch.eye(len(MONO), dtype=A.dtype, device=A.device))
    D = torch.diagonal(A, dim1=1, dim2=2).detach().rsqrt()
    L, info = torch.linalg.cholesky_ex(A * D[:, :, None] * D[:, None, :])
    ok = ok & (info == 0)  # a fit without a factorisation counts as singular: zero derivatives

    def solve(b):
        y = torch.linalg.solve_triangular(L, D[:, :, None] * b, upper=False)
        return D[:, :, None] * torch.linalg.solve_triangular(L.transpose(1, 2), y, upper=True)

    c = solve(WP.transpose(1, 2) @ du)
    for _ in range(refine):
        c = c + solve(WP.transpose(1, 2) @ (du - P @ c))
    c = torch.where(ok[:, None, None], c, 0.0).permute(2, 1, 0)
    twice = torch.tensor([2.0, 1.0, 1.0, 2.0, 1.0, 2.0], dtype=c.dtype, device=c.device)
    return c[:, LIN] / lam[i], c[:, QUAD] * twice[None, :, None] / lam[i] ** 2


def _rhs_of(u, g, h, lam, gamma, laws):
    rho, V, B, sig = u[0], u[1:4], u[4:7], u[7]
    gV, gB, div = g[1:4], g[4:7], g[1, 0] + g[2, 1] + g[3, 2]
    zeta = eta = torch.zeros_like(rho)
    if laws:
        cf = ((gamma * (gamma - 1.0) * sig + (B * B).sum(0)) / rho).sqrt()
        zeta = laws["c_zeta_l"] * lam * cf + laws["c_zeta_a"] * lam ** 2 * (-div).clamp(min=0.0)
        eta = laws["c_eta"] * lam * cf
    J = torch.stack([gB[2, 1] - gB[1, 2], gB[0, 2] - gB[2, 0], gB[1, 0] - gB[0, 1]])
    force = torch.cross(J, B, dim=0) - (gamma - 1.0) * g[7]
    gdivV = torch.stack([sum(h[1 + c, HESS[a][c]] for c in range(3)) for a in range(3)])
    gdivB = torch.stack([sum(h[4 + c, HESS[a][c]] for c in range(3)) for a in range(3)])
    dV = force / rho + zeta * gdivV
    dB = (gV * B[None]).sum(1) - B * div + eta * gdivB
    return torch.cat([(-rho * div)[None], dV, dB, (-gamma * sig * div + rho * zeta * div * div)[None]])


def _parts(lists):
    n = lists[0].numel() - 1
    size = 1 << 14
    return [torch.arange(a, min(a + size, n), device=lists[0].device) for a in range(0, n, size)]


def _rhs(box, pos, lam, U, lists, gamma, laws=None, refine=2):
    out = torch.empty_like(U)
    for i in _parts(lists):
        g, h = _fit(box, pos, lam, U, lists, i, refine)
        out[:, i] = _rhs_of(U[:, i], g, h, lam[i], gamma, laws)
    return out


def _heun(box, pos, lam, U, gamma, dt, frozen):
    laws = LAWS if frozen is not None else None
    h = torch.full_like(lam, dt) if frozen is None else torch.where(frozen, 0.0, dt)
    F0 = _rhs(box, pos, lam, U, _lists(box, pos, lam), gamma, laws)
    p1, U1 = pos + h * U[1:4], U + h * F0
    F1 = _rhs(box, p1, lam, U1, _lists(box, p1, lam), gamma, laws)
    return pos + 0.5 * h * (U[1:4] + U1[1:4]), U + 0.5 * h * (F0 + F1)


def _levels(box, pos, lam, U, gamma, dt_max, most):
    P = (gamma - 1.0) * U[7]
    c2 = (gamma * P + ((U[4] * U[4] + U[5] * U[5]) + U[6] * U[6])) / U[0]
    dt = CFL * lam / c2.sqrt()
    L0 = torch.zeros_like(lam, dtype=torch.int64)
    for k in range(most):
        L0 = torch.where((L0 == k) & (dt_max / 2 ** k > dt), k + 1, L0)
    off, mem = _lists(box, pos, lam)
    send = torch.repeat_interleave(L0 - 1, off[1:] - off[:-1])
    return L0.scatter_reduce(0, mem, send, "amax", include_self=True)


def _block(box, pos, lam, U, gamma):
    """One synchronised step of individual power-of-two steps (two levels below the coarsest)."""
    dt_max, most = _dt_max(lam, U, gamma), 2
    lv = _levels(box, pos, lam, U, gamma, dt_max, most)
    m, delta = 2 ** (most - lv), dt_max / 2 ** most
    F = _rhs(box, pos, lam, U, _lists(box, pos, lam), gamma, refine=1)
    ax, aU, aF = pos, U, F
    for k in range(2 ** most):
        tau = (k + 1 - (k // m) * m) * delta
        pos, U = ax + tau * aU[1:4], aU + tau * aF
        ends = (k + 1) % m == 0
        F = _rhs(box, pos, lam, U, _lists(box, pos, lam), gamma, refine=1)
        half = 0.5 * m * delta
        pos, U = (torch.where(ends, ax + half * (aU[1:4] + U[1:4]), pos), torch.where(ends, aU + half * (aF + F), U))
        ax, aU = torch.where(ends, pos, ax), torch.where(ends, U, aU)
        F = _rhs(box, pos, lam, U, _lists(box, pos, lam), gamma, refine=1)
        aF = torch.where(ends, F, aF)
    return pos, U


def _candidates(box, pos, lam):
    """Places for new particles: the void point of each particle farthest from its neighbours."""
    lists = _lists(box, pos, lam)
    cand = torch.zeros_like(pos)
    for i in _parts(lists):
        j, there = _padded(lists, i)
        d = _offset(box, pos[:, j] - pos[:, i, None])
        r = RF * lam[i]
        h, dv2, rin = 0.25 * r, (VOID * lam[i]) ** 2, r - VOID * lam[i]
        far = torch.full_like(r, -1.0)
        place = torch.zeros((3, i.numel()), dtype=pos.dtype, device=pos.device)
        for kx in range(-4, 5):
            for ky in range(-4, 5):
                for kz in range(-4, 5):
                    if kx * kx + ky * ky + kz * kz > 6:
                        continue
                    o = torch.stack([kx * h, ky * h, kz * h])
                    o2 = _square(o)
                    e2 = torch.where(there, _square(d - o[:, :, None]), math.inf).amin(1)
                    clear = torch.minimum(e2, o2)
                    take = (o2 < rin * rin) & ~(o2 < dv2) & ~(e2 < dv2) & (clear > far)
                    far = torch.where(take, clear, far)
                    place = torch.where(take, pos[:, i] + o, place)
        cand[:, i] = place
    return cand


def exact(case, seed):
    kind, n = case["kind"], _count(case)
    if kind == "host" or n > 1_100_000:
        return None  # the host step's state is in the library's storage order; over a million takes too long
    if kind == "eager" and not case.get("open", False):
        return None  # storage order again
    if kind == "block" and n > 250_000:
        return None
    box, pos, lam, U, gamma, dt, _, frozen, gbar = _inputs(case, seed)
    if kind in ("step", "eager"):
        return _heun(box, pos, lam, U, gamma, dt, frozen)
    if kind == "block":
        return (*_block(box, pos, lam, U, gamma), None)
    if kind == "scan":
        return None, None, _candidates(box, pos, lam), None, None
    lists = _lists(box, pos, lam)
    if kind == "rhs64":
        return _rhs(box, pos, lam, U, lists, gamma)
    if kind == "derivs64":
        g, h = zip(*(_fit(box, pos, lam, U, lists, i, 2) for i in _parts(lists)))
        return torch.cat(g, 2), torch.cat(h, 2), None
    out = _rhs(box, pos, lam, U, lists, gamma)
    pos.requires_grad_(True)
    U.requires_grad_(True)
    for i in _parts(lists):
        g, h = _fit(box, pos, lam, U, lists, i, 0)
        (_rhs_of(U[:, i], g, h, lam[i], gamma, None) * gbar[:, i]).sum().backward()
    return out, pos.grad, U.grad
