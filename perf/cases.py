"""Performance cases of the LELBM time step: what a user of this library has it do.

A case is one pass through the public entry points on a state that the user has in hand on the
device: the moments go in (lelbm_set_moments_device), a few steps run, the moments come out
(lelbm_get_moments_device).  Handles, warm-start networks and buffers are kept between passes, as
a solver's main loop keeps them.  The states are developed flows, not initial conditions: fronts a
few cells wide with the non-equilibrium moments that belong to them, near-equilibrium elsewhere.

`exact` restates the step in plain torch in FP64: every cell's velocity set as an explicit list.
"""
from __future__ import annotations

import math
import os

import numpy as np
import torch

from paper_2508_06911_gb300 import lelbm as L
from paper_2508_06911_gb300 import workloads as W
from paper_2508_06911_gb300.solver import Solver

GAMMA = 1.4
PRANDTL = 0.71
PRECISION = {"fp64": L.LELBM_FP64, "mixed": L.LELBM_MIXED, "fp32": L.LELBM_FP32}
WEIGHTS = os.path.join(os.path.dirname(os.path.abspath(L.__file__)), "weights")
N_MOM = {1: 6, 2: 11, 3: 17}
N_F = {1: 4, 2: 10, 3: 19}
N_G = {1: 3, 2: 6, 3: 10}


def listed():
    return [
        # the smallest problem: one 400-cell Riemann tube, where launches and latency are the time
        dict(name="tube_400_fp64", kind="tube", n=400, precision="fp64", steps=8),
        # a parameter study: 4096 tubes of 256 to 4096 cells in one persistent launch, at full tolerance
        dict(name="batch_4096_mixed", kind="batch", tubes=4096, precision="mixed", start="maxwell", steps=2),
        # the same study in single precision with the learned start
        dict(name="batch_4096_fp32", kind="batch", tubes=4096, precision="fp32", start="learned", steps=1),
        # the reference-grade FP64 path on a ragged rectangle with outflow pads
        dict(name="flow_731x523_fp64", kind="flow", nx=731, ny=523, precision="fp64", start="maxwell", steps=1,
             RT_hi=1.5, umax=1.5, periodic=False),
        # the benchmark's own grid and path: production runs of the four-quadrant problem
        dict(name="flow_4096_mixed", kind="flow", nx=4096, ny=4096, precision="mixed", start="learned", steps=1,
             RT_hi=1.5, umax=1.5, periodic=False),
        # single precision from the Maxwellian start, a mid-size production grid
        dict(name="flow_2048_fp32", kind="flow", nx=2048, ny=2048, precision="fp32", start="maxwell", steps=1,
             RT_hi=1.5, umax=1.5, periodic=False),
        # hot gas moving ten cells a step: velocity sets of hundreds of points
        dict(name="hotbox_512_mixed", kind="flow", nx=512, ny=512, precision="mixed", start="maxwell", steps=1,
             RT_lo=7.0, RT_hi=9.0, umax=0.5, drift=10.0, periodic=True),
        # supersonic flow past a slip-wall cylinder: inflow, outflow and traced walls
        dict(name="cylinder_1024x512_mixed", kind="cylinder", nx=1024, ny=512, precision="mixed", start="maxwell",
             steps=1),
        # three dimensions, FP64
        dict(name="flow3d_40_fp64", kind="flow3d", n=40, precision="fp64", steps=1, RT_hi=1.0, umax=1.0),
        # runs that must repeat bit by bit: the fixed-order gather
        dict(name="flow_384x320_deterministic", kind="flow", nx=384, ny=320, precision="fp64", start="maxwell",
             steps=1, RT_hi=1.5, umax=1.5, periodic=False, deterministic=True),
        # an application that owns its memory: one step on its own buffers
        dict(name="noalloc_257x193_fp64", kind="noalloc", nx=257, ny=193, precision="fp64", steps=1, RT_hi=1.5,
             umax=1.5),
        # training the learned start: loss and gradient over the pairs of one 1024 x 1024 step
        dict(name="pairs_1m", kind="pairs", dims=2, pairs=1 << 20),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["tube", "batch", "batch", "flow", "flow", "flow", "flow", "hot", "cylinder", "flow3d",
                       "deterministic", "noalloc", "pairs"])
    steps = rng.choice([1, 1, 2, 3])
    if kind == "tube":
        return dict(kind="tube", n=_log(rng, 64, 4096), precision=rng.choice(["fp64", "mixed"]),
                    steps=rng.randint(1, 16))
    if kind == "batch":
        p = rng.choice(["fp64", "mixed", "fp32"])
        return dict(kind="batch", tubes=_log(rng, 48, 1024 if p == "fp64" else 4096), precision=p,
                    start=rng.choice(["maxwell", "learned"]), steps=1 if p == "fp32" else rng.randint(1, 2))
    if kind == "flow":
        p = rng.choice(["fp64", "mixed", "fp32"])
        hi = 700 if p == "fp64" else 2048
        return dict(kind="flow", nx=_log(rng, 48, hi), ny=_log(rng, 48, hi), precision=p,
                    start=rng.choice(["maxwell", "learned"]), steps=1 if p == "fp32" else rng.choice([1, 1, 2]),
                    RT_hi=round(math.exp(rng.uniform(math.log(0.5), math.log(4.0))), 3),
                    umax=round(rng.uniform(0.3, 2.0), 3), periodic=rng.random() < 0.3)
    if kind == "hot":
        RT = math.exp(rng.uniform(math.log(0.5), math.log(24.0)))
        return dict(kind="flow", nx=_log(rng, 64, 512), ny=_log(rng, 64, 512), precision=rng.choice(["mixed", "fp32"]),
                    start="maxwell", steps=1, RT_lo=round(0.85 * RT, 3), RT_hi=round(1.15 * RT, 3), umax=0.5,
                    drift=float(rng.randint(0, 12)), periodic=True)
    if kind == "cylinder":
        ny = _log(rng, 96, 768)
        return dict(kind="cylinder", nx=2 * ny + rng.randint(0, 5), ny=ny, precision=rng.choice(["mixed", "fp64"])
                    if ny < 256 else "mixed", start=rng.choice(["maxwell", "learned"]), steps=1)
    if kind == "flow3d":
        return dict(kind="flow3d", n=_log(rng, 10, 40), precision="fp64", steps=1,
                    RT_hi=round(rng.uniform(0.4, 1.2), 3), umax=round(rng.uniform(0.2, 1.5), 3))
    if kind == "deterministic":
        return dict(kind="flow", nx=_log(rng, 48, 400), ny=_log(rng, 48, 400), precision="fp64", start="maxwell",
                    steps=steps, RT_hi=round(rng.uniform(0.5, 2.0), 3), umax=round(rng.uniform(0.3, 2.0), 3),
                    periodic=rng.random() < 0.5, deterministic=True)
    if kind == "noalloc":
        return dict(kind="noalloc", nx=_log(rng, 48, 500), ny=_log(rng, 48, 500), precision="fp64", steps=1,
                    RT_hi=round(rng.uniform(0.5, 2.0), 3), umax=round(rng.uniform(0.3, 2.0), 3))
    return dict(kind="pairs", dims=rng.choice([1, 2]), pairs=_log(rng, 1 << 12, 1 << 20))


# ---------------------------------------------------------------------------
# States
# ---------------------------------------------------------------------------
def _generator(seed, tag):
    return np.random.Generator(np.random.PCG64([seed & 0x7FFFFFFF, tag]))


class _Waves:
    """Smooth random fields in [-1, 1] on coordinates x[a] in [0, 1): three Fourier modes each."""

    def __init__(self, g, x):
        self.g, self.x = g, x

    def __call__(self):
        f = 0.0
        for _ in range(3):
            k = self.g.integers(-2, 3, len(self.x))
            p = 2 * math.pi * self.g.random()
            f = f + torch.cos(sum(2 * math.pi * int(ka) * xa for ka, xa in zip(k, self.x)) + p)
        return f / 3.0


def _moments(rho, u, RT, K, eps, wave):
    """Raw moments of a gas at (rho, u, RT) with non-equilibrium parts of relative size eps."""
    D = len(u)
    P = [[None] * D for _ in range(D)]
    for a in range(D):
        for b in range(a, D):
            P[a][b] = P[b][a] = rho * RT * eps * wave()
    trP = sum(P[a][a] for a in range(D))
    s = RT.sqrt()
    usq = sum(v * v for v in u)
    G0 = rho * K * RT - trP
    M = [rho] + [rho * v for v in u]
    M += [rho * u[a] * u[b] + (rho * RT if a == b else 0.0) + P[a][b] for a in range(D) for b in range(a, D)]
    M += [rho * (usq + (D + 2) * RT) * u[c] + 2 * sum(u[a] * P[a][c] for a in range(D)) + u[c] * trP
          + rho * RT * s * eps * wave() for c in range(D)]
    M += [G0] + [u[c] * G0 + rho * RT * s * eps * wave() for c in range(D)]
    return torch.stack([m.expand_as(rho) for m in M])


def _flow_interior(shape, seed, RT_lo, RT_hi, umax, drift, periodic):
    """Moments [n_mom, *shape] of a flow of 2^D regions: temperatures log-uniform in [RT_lo, RT_hi]
    (both met), densities in [0.1, 1.5], velocities up to umax (plus a drift per axis), wavy fronts
    two cells wide (periodic flows have a second front at the wrap)."""
    D = len(shape)
    g = _generator(seed, 11 + D)
    ax = [torch.arange(n, dtype=torch.float64, device="cuda") for n in reversed(shape)]  # x, y[, z] cell indices
    idx = [a.view([-1 if d == D - 1 - k else 1 for d in range(D)]) for k, a in enumerate(ax)]
    x = [(i + 0.5) / n for i, n in zip(idx, reversed(shape))]
    side, front = [], 0.0
    for a in range(D):
        n = shape[D - 1 - a]
        others = [x[b] for b in range(D) if b != a]
        bend = 0.04 * sum(torch.sin(2 * math.pi * (o + g.random())) for o in others)
        s = 0.5 * (1 + torch.tanh((x[a] - 0.5 - bend) * n / 2.0))
        if periodic:
            s = s * 0.5 * (1 - torch.tanh((x[a] - 0.92) * n / 2.0))
        side.append(s)
        front = torch.maximum(front, 4 * s * (1 - s)) if a else 4 * s * (1 - s)
    n_reg = 2 ** D
    T = RT_lo * (RT_hi / RT_lo) ** g.random(n_reg)
    T[g.permutation(n_reg)[:2]] = RT_lo, RT_hi
    R = g.uniform(0.1, 1.5, n_reg)
    V = g.standard_normal((n_reg, D))
    V *= (umax * g.random(n_reg) ** (1.0 / D) / np.linalg.norm(V, axis=1))[:, None]

    def blend(v):
        out = 0.0
        for k in range(n_reg):
            w = float(v[k])
            for a in range(D):
                w = w * (side[a] if (k >> a) & 1 else 1 - side[a])
            out = out + w
        return out

    wave = _Waves(g, x)
    rho = blend(R) * (1 + 0.02 * wave())
    RT = blend(T) * (1 + 0.01 * wave()).clamp(min=1.0)
    u = [blend(V[:, a]) + drift + 0.02 * wave() for a in range(D)]
    rho, RT = rho.expand(shape), RT.expand(shape)
    u = [v.expand(shape) for v in u]
    return _moments(rho, u, RT, W.internal_dof(GAMMA, D), (1e-4 + 0.04 * front).expand(shape), wave)


def _flow_args(case):
    D = 3 if case["kind"] == "flow3d" else 2
    shape = (case["n"],) * 3 if D == 3 else (case["ny"], case["nx"])
    a = dict(RT_lo=case.get("RT_lo", 0.25), RT_hi=case["RT_hi"], umax=case["umax"], drift=case.get("drift", 0.0),
             periodic=case.get("periodic", True))
    pad = 0 if a["periodic"] else W.pad_for(1.3 * a["umax"] + abs(a["drift"]), 1.5 * a["RT_hi"])
    return D, shape, pad, a


def _padded(m, pad):
    return torch.nn.functional.pad(m, (pad,) * (2 * (m.dim() - 1))) if pad else m


def _cylinder(case):
    """(solid mask [ny, nx], lattice inflow velocity, RT of the stream, pad): Mach 3, slip wall."""
    nx, ny = case["nx"], case["ny"]
    RT, mach = 0.5, 3.0
    u = mach * math.sqrt(GAMMA * RT)
    X, Y = np.meshgrid(np.arange(nx) + 0.5, np.arange(ny) + 0.5)
    solid = ((X - nx / 4) ** 2 + (Y - ny / 2) ** 2 <= (ny / 16) ** 2).astype(np.uint8)
    return solid, u, RT, W.pad_for(1.3 * u, RT * (1 + 0.2 * mach * mach) * 1.5)


def _tubes(case, seed):
    """Layout and moments of a batch of tubes (or one): blended two-state problems, acoustic scaling.
    The layout is the case's; the seed varies every tube's states."""
    w = W.riemann_1d(case["n"]) if case["kind"] == "tube" else W.riemann_1d_batch(case["tubes"])
    dev = dict(dtype=torch.float64, device="cuda")
    n, p = (torch.as_tensor(np.asarray(v), device="cuda") for v in (w.lengths, w.pads))
    tot = n + 2 * p
    first = torch.cumsum(tot, 0) - tot
    inst = torch.repeat_interleave(torch.arange(len(tot), device="cuda"), tot)
    i = torch.arange(int(tot.sum()), device="cuda") - first[inst] - p[inst]
    inside = (i >= 0) & (i < n[inst])
    x = (i + 0.5) / n[inst]
    s = 0.5 * (1 + torch.tanh((x - 0.5) * n[inst] / 2.0))
    lt, rt, sc = (torch.as_tensor(np.asarray(v), **dev)[inst] for v in (w.left, w.right, w.scale))
    g = _generator(seed, 7)
    wave = _Waves(g, [x])
    f = [torch.as_tensor(g.uniform(a, b, len(tot)), **dev)[inst] for a, b in ((0.8, 1.25), (0.9, 1.0), (1.0, 1.2))]
    rho = (lt[:, 0] * (1 - s) + rt[:, 0] * s) * f[0] * (1 + 0.02 * wave())
    u = (lt[:, 1] * (1 - s) + rt[:, 1] * s) * sc * f[1]
    RT = (lt[:, 2] / lt[:, 0] * (1 - s) + rt[:, 2] / rt[:, 0] * s) * sc * sc * f[2]
    M = _moments(rho, [u], RT, w.K, 1e-4 + 0.04 * 4 * s * (1 - s), wave)
    return w, (M * inside).contiguous(), (inst, first + p, n, p)


def _network(dims, seed):
    """Parameters of a warm-start network to be trained, and feature/target pairs like recorded ones."""
    nin, nout, total, n_weights = L.lelbm_mlp_size(dims)
    return nin, nout, total, n_weights, torch.Generator(device="cuda").manual_seed(seed)


def _pairs(case, seed):
    nin, nout, _, n_w, g = _network(case["dims"], seed)
    dev = dict(device="cuda", generator=g)
    X = torch.randn(case["pairs"], nin, **dev) * 0.3 + torch.linspace(-0.5, 1.5, nin, device="cuda")
    mix = torch.randn(nin, nout, **dev) / nin ** 0.5
    Y = 0.05 * torch.tanh(X @ mix) + 0.005 * torch.randn(case["pairs"], nout, **dev)
    parts = []
    for rows, cols, gain in ((64, nin, 1.0), (64, 64, 1.0), (nout, 64, 0.5)):
        parts += [(torch.rand(rows * cols, **dev) * 2 - 1) * gain * (6.0 / cols) ** 0.5,
                  (torch.rand(rows, **dev) * 2 - 1) * 0.1]
    params = torch.cat(parts + [X.mean(0), X.std(0), Y.mean(0), Y.std(0)]).float().contiguous()
    return params, X.contiguous(), Y.contiguous(), n_w


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.kind, s.case = case["kind"], case
    s.stream = torch.cuda.Stream()
    raw = s.stream.cuda_stream
    if s.kind == "pairs":
        s.params, s.X, s.Y, n_w = _pairs(case, seed)
        s.grad = torch.empty(n_w, device="cuda")
        return s
    prec = PRECISION[case["precision"]]
    if s.kind in ("tube", "batch"):
        w, s.M, _ = _tubes(case, seed)
        many = w.n_batch > 1
        s.solver = Solver(1, int(w.lengths[0]), K=w.K, nu=w.nu, Pr=w.Pr, bc=(0, 0, 2, 2), pad=int(w.pads[0]),
                          lengths=w.lengths if many else None, pads=w.pads if many else None, stream=raw,
                          precision=prec)
    elif s.kind == "cylinder":
        solid, u, RT, pad = _cylinder(case)
        M = _flow_interior((case["ny"], case["nx"]), seed, RT, 1.2 * RT, 0.2, 0.0, False)
        D2 = W.internal_dof(GAMMA, 2)
        # the stream: boost every cell's state by the inflow velocity
        rho, ux, uy = M[0], M[1] / M[0], M[2] / M[0]
        T = ((M[3] + M[5] + M[8]) / rho - ux * ux - uy * uy) / (2 + D2)
        g = _generator(seed, 29)
        x = [(torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) / n for n in (case["nx"], case["ny"])]
        wave = _Waves(g, [x[0][None, :], x[1][:, None]])
        M = _moments(rho * 2, [ux + u, uy], T, D2, torch.full_like(rho, 5e-3), wave)
        s.M = _padded(M * torch.as_tensor(1.0 - solid, device="cuda"), pad).contiguous()
        s.solver = Solver(2, case["nx"], case["ny"], K=D2, nu=0.0, Pr=PRANDTL, bc=(1, 0, 0, 0), pad=pad,
                          solid=np.pad(solid, pad).reshape(-1), inlet=(1.4, u, 0.0, RT), stream=raw, precision=prec)
    elif s.kind in ("flow", "flow3d", "noalloc"):
        D, shape, pad, a = _flow_args(case)
        s.M = _padded(_flow_interior(shape, seed, **a), pad).contiguous()
        K = W.internal_dof(GAMMA, D)
        bc = (2 if a["periodic"] else 0,) * (6 if D == 3 else 4)
        if s.kind == "noalloc":
            p = L.lelbm_default_params()
            p.dims, p.nx, p.ny, p.pad, p.K, p.nu_shear, p.prandtl = 2, shape[1], shape[0], pad, K, 1e-3, PRANDTL
            p.precision, p.stream = prec, raw
            for k in range(4):
                p.bc[k] = bc[k]
            s.params, s.out = p, torch.empty_like(s.M)
            return s
        s.solver = Solver(D, shape[-1], shape[-2], nz=shape[0] if D == 3 else 1, K=K, nu=1e-3, Pr=PRANDTL, bc=bc,
                          pad=pad, stream=raw, precision=prec, deterministic=int(case.get("deterministic", False)))
    if case.get("start") == "learned":
        net = "warmstart_1d.npy" if s.solver.dims == 1 else "warmstart_2d_quadrants.npy"
        L.lelbm_set_mlp(s.solver.h, np.load(os.path.join(WEIGHTS, net)))
        L.lelbm_set_mlp_gate(s.solver.h, 1e-3)
    s.out = torch.empty_like(s.M)
    return s


def run(s):
    if s.kind == "pairs":
        loss = L.lelbm_mlp_loss_grad(s.case["dims"], s.params.data_ptr(), s.X.data_ptr(), s.Y.data_ptr(),
                                     s.X.shape[0], s.grad.data_ptr(), s.stream.cuda_stream)
        return {"loss": loss, "grad": s.grad}
    if s.kind == "noalloc":
        L.lelbm_step_noalloc(s.params, s.M.data_ptr(), s.out.data_ptr())
        return s.out
    h = s.solver.h
    L.lelbm_set_moments_device(h, s.M.data_ptr())
    if s.kind == "batch":
        s.solver.run_batch(s.case["steps"])
    else:
        s.solver.step(s.case["steps"])
    L.lelbm_get_moments_device(h, s.out.data_ptr())
    if s.case["precision"] == "fp32":  # the single-precision path's user keeps single-precision fields
        with torch.cuda.stream(s.stream):
            return s.out.float()
    return s.out


def work(case):
    """Each moment read and written once per step; per cell the collision, two Newton updates and the
    check after them, and the streaming pass, over the mean size of the velocity set."""
    if case["kind"] == "pairs":
        nin, nout, _, n_w = L.lelbm_mlp_size(case["dims"])
        return {"bytes": 4.0 * case["pairs"] * (nin + nout) + 8.0 * n_w, "flops": 6.0 * case["pairs"] * n_w}
    D = {"tube": 1, "batch": 1, "flow3d": 3}.get(case["kind"], 2)
    lo, hi = case.get("RT_lo", 0.25), case.get("RT_hi", 6.0 if case["kind"] == "batch" else 1.5)
    q = 0.0
    for k in range(16):  # temperatures log-uniform between the coldest and the hottest region
        r = max(2, math.floor(4 * math.sqrt(lo * (hi / lo) ** ((k + 0.5) / 16)) + 0.5)) + 0.5
        q += {1: 2 * r, 2: math.pi * r * r, 3: 4 / 3 * math.pi * r ** 3}[D] / 16
    cells = {"tube": lambda: case["n"], "batch": lambda: 1384.0 * case["tubes"],
             "flow3d": lambda: case["n"] ** 3}.get(case["kind"], lambda: case["nx"] * case["ny"])()
    cells *= case.get("steps", 1)
    per_point = 3 * (6 + 2 * 7 + 6 + 4 + 2 * 5) + 2 * N_MOM[D] + 10
    solve = sum(n ** 3 / 3.0 + 2.0 * n * n for n in (N_F[D], N_G[D]))
    return {"bytes": 16.0 * N_MOM[D] * cells, "flops": cells * (q * per_point + 2 * solve + 200.0)}


# ---------------------------------------------------------------------------
# The step in plain FP64 torch
# ---------------------------------------------------------------------------
def _pair_list(D):
    return [(a, b) for a in range(D) for b in range(a, D)]


def _exact_collision(M, D, K, nu):
    """rho, u, RT and the constraints in thermal units (fluons, phonons) of moments M [n_mom, n]."""
    pos = {p: 1 + D + k for k, p in enumerate(_pair_list(D))}
    second = lambda a, b: M[pos[(min(a, b), max(a, b))]]  # noqa: E731
    i_md = 1 + D + len(pos)
    i_g = i_md + D
    rho = M[0]
    u = [M[1 + a] / rho for a in range(D)]
    usq = sum(v * v for v in u)
    RT = ((sum(second(a, a) for a in range(D)) + M[i_g]) / rho - usq) / (D + K)
    s = RT.sqrt()
    P = [[second(a, b) - rho * (u[a] * u[b] + (RT if a == b else 0.0)) for b in range(D)] for a in range(D)]
    trP = sum(P[a][a] for a in range(D))
    Q = [M[i_md + c] - 2 * sum(u[a] * P[a][c] for a in range(D)) - u[c] * trP - rho * (usq + (D + 2) * RT) * u[c]
         for c in range(D)]
    G0n = M[i_g] - rho * K * RT
    Gn = [M[i_g + 1 + c] - u[c] * M[i_g] for c in range(D)]
    inv_f = nu / RT + 0.5
    w = [1 / inv_f, torch.ones_like(RT), 1 / ((inv_f - 0.5) / PRANDTL + 0.5)]
    k2 = (sum(abs(P[a][b]) for a in range(D) for b in range(D)) + abs(G0n)) / rho / ((D + K) * RT)
    k3 = (sum(abs(v) for v in Q) + sum(abs(v) for v in Gn)) / rho / ((D + K + 2) * RT * s)
    x = (torch.log10(torch.maximum(k2, k3).clamp(min=1e-30)) + 2).clamp(0.0, 1.0)
    wf, wb, wh = (v + (1 - v) * x for v in w)
    bulk = -G0n / D
    one, zero = torch.ones_like(RT), torch.zeros_like(RT)
    cf = [one] + [zero] * D
    for a, b in _pair_list(D):
        d = 1.0 if a == b else 0.0
        cf.append((d * rho * RT + (1 - wf) * (P[a][b] - d * bulk) + (1 - wb) * d * bulk) / (rho * RT))
    cf += [(1 - wh) * (1 + 2 * (a == c)) / (D + 2) * Q[c] / (rho * RT * s) for c in range(D) for a in range(D)]
    nrm = rho * K * RT
    cg = [(nrm + (1 - wb) * G0n) / nrm] + [(1 - wh) * v / (nrm * s) for v in Gn]
    cg += [one if a == b else zero for a, b in _pair_list(D)]
    return rho, torch.stack(u, 1), RT, torch.stack(cf, 1), torch.stack(cg, 1)


def _basis(t, fluon):
    D = t.shape[-1]
    v = [torch.ones_like(t[..., 0])] + [t[..., a] for a in range(D)]
    v += [t[..., a] * t[..., b] for a, b in _pair_list(D)]
    if fluon:
        v += [t[..., a] * t[..., a] * t[..., c] for c in range(D) for a in range(D)]
    return torch.stack(v, -1)


def _velocity_set(u, R, levels, D):
    """Points [n, q, D], weights [n, q] (0 for a point that is not in a cell's set) and how many of
    the q are on the lattice; the rest are refined children."""
    dev = u.device

    def offsets(lo, hi):
        k = torch.arange(lo, hi + 1, dtype=torch.float64, device=dev)
        return torch.stack(torch.meshgrid(*([k] * D), indexing="ij"), -1).reshape(-1, D)

    def dist2(c):
        d = c - u[:, None, :]
        return (d * d).sum(-1)

    base = u.floor()[:, None, :]
    c = base + offsets(-R - 1, R + 2)
    d2 = dist2(c)
    inside = d2 <= (R + 0.5) ** 2
    pts, wts = [c], [(inside & ~(d2 <= 2.25) if levels else inside).double()]
    if levels:
        c = base + offsets(-2, 3)
        d2 = dist2(c)
        split = (d2 <= (R + 0.5) ** 2) & (d2 <= 2.25)
        for lv in range(1, levels + 1):
            h = 0.5 ** (lv - 1)
            kid = (offsets(0, 1) - 0.5) * (0.5 * h)
            c = (c[:, :, None, :] + kid).reshape(c.shape[0], -1, D)
            member = split.repeat_interleave(2 ** D, 1)
            again = member & (dist2(c) <= (3 * 0.5 ** (lv + 1)) ** 2) if lv < levels else torch.zeros_like(member)
            pts.append(c)
            wts.append((member & ~again).double() * 0.5 ** (D * lv))
            split = again
    return torch.cat(pts, 1), torch.cat(wts, 1), pts[0].shape[1]


def _multipliers(t, w, con, RT, fluon):
    """Newton on the multipliers until the residual is at rounding; populations [n, q]."""
    D = t.shape[-1]
    T = _basis(t, fluon)
    lam = torch.zeros_like(con)
    lam[:, 0] = -1 + 0.5 * D * torch.log(2 * math.pi * RT)
    for k, (a, b) in enumerate(_pair_list(D)):
        if a == b:
            lam[:, 1 + D + k] = 0.5
    last = False
    for _ in range(30):
        f = torch.where(w > 0, w * torch.exp(-1 - (T @ lam[:, :, None])[..., 0]), 0.0)
        if last:
            break
        Tf = T * f[..., None]
        r = Tf.sum(1) - con
        lam = lam + torch.linalg.solve(T.transpose(1, 2) @ Tf, r)
        last = float(r.abs().max()) <= 1e-13 or (_ > 8 and float(r.abs().max()) <= 1e-12)
    return f


def _exact_step(M, D, K, nu, index, extent, periodic, stride, origin):
    """One step.  index[a]: interior coordinate of every cell along axis a (negative or beyond on
    pads); extent[a]: interior cells; origin: linear index of interior coordinate 0."""
    n_cell = M.shape[1]
    out = torch.zeros_like(M)
    rho, u, RT, cf, cg = _exact_collision(M, D, K, nu)
    sig = RT.sqrt()
    R = torch.floor(4 * sig + 0.5).clamp(min=2).long()
    lv = torch.floor(1 / (3 * sig) + 0.5).clamp(max=4).long()
    key = R * 8 + lv
    for kk in torch.unique(key).tolist():
        r, levels = kk // 8, kk % 8
        q = (2 * r + 4) ** D + (sum(6 ** D * 2 ** (D * k) for k in range(1, levels + 1)))
        which = torch.nonzero(key == kk)[:, 0]
        chunk = max(1, 400_000_000 // (8 * q * (N_F[D] + 6)))
        for sel in which.split(chunk):
            pts, w, n0 = _velocity_set(u[sel], r, levels, D)
            t = (pts - u[sel][:, None, :]) / sig[sel][:, None, None]
            f = _multipliers(t, w, cf[sel], RT[sel], True) * rho[sel][:, None]
            g = _multipliers(t, w, cg[sel], RT[sel], False) * (rho * K * RT)[sel][:, None]
            for part, shares in ((slice(0, n0), 1), (slice(n0, None), 2 ** D)):
                c = pts[:, part]
                if c.shape[1] == 0:
                    continue
                fl = c.floor()
                fr = c - fl
                val = [f[:, part] * T for T in _basis(c, True).unbind(-1)[: 1 + D + D * (D + 1) // 2]]
                csq = (c * c).sum(-1)
                val += [f[:, part] * csq * c[..., a] for a in range(D)]
                val += [g[:, part]] + [g[:, part] * c[..., a] for a in range(D)]
                for k in range(shares):
                    wgt = (w[:, part] > 0).double()
                    tgt = torch.zeros_like(fl[..., 0]).long() + (origin[sel][:, None] if torch.is_tensor(origin) else origin)
                    ok = w[:, part] > 0
                    for a in range(D):
                        up = (k >> a) & 1
                        wgt = wgt * (fr[..., a] if up else 1 - fr[..., a])
                        at = index[a][sel][:, None] + fl[..., a].long() + up
                        ext = extent[a][sel][:, None] if torch.is_tensor(extent[a]) else extent[a]
                        if periodic:
                            at = at % ext
                        else:
                            ok = ok & (at >= 0) & (at < ext)
                        tgt = tgt + at * stride[a]
                    tgt = tgt[ok]
                    for m in range(N_MOM[D]):
                        out[m].index_add_(0, tgt, (val[m] * wgt)[ok])
    return out


def _exact_pairs(case, seed):
    params, X, Y, n_w = _pairs(case, seed)
    nin, nout = X.shape[1], Y.shape[1]
    wts = params[:n_w].bfloat16().double()  # the network's weights are BF16; all arithmetic in FP64
    nrm = params[n_w:].double()
    W1, b1, W2, b2, W3, b3 = wts.split([64 * nin, 64, 64 * 64, 64, nout * 64, nout])
    xm, xs, ym, ys = nrm.split([nin, nin, nout, nout])
    p = [v.clone().requires_grad_() for v in (W1, b1, W2, b2, W3, b3)]
    total = 0.0
    for x, y in zip(X.split(1 << 18), Y.split(1 << 18)):
        h = torch.nn.functional.silu((x.double() - xm) / xs @ p[0].view(64, nin).T + p[1])
        h = torch.nn.functional.silu(h @ p[2].view(64, 64).T + p[3])
        e = h @ p[4].view(nout, 64).T + p[5] - (y.double() - ym) / ys
        part = (e * e).sum() / (X.shape[0] * nout)
        part.backward()
        total += float(part)
    return {"loss": total, "grad": torch.cat([v.grad for v in p])}


def exact(case, seed):
    kind = case["kind"]
    if kind == "pairs":
        return _exact_pairs(case, seed)
    if kind == "cylinder":  # its walls are traced path by path: no plain form, and minutes in Python
        return None
    if kind in ("tube", "batch"):
        w, M, (inst, lo, n, p) = _tubes(case, seed)
        i = torch.arange(M.shape[1], device="cuda") - lo[inst]
        src = i.clamp(min=0).minimum(n[inst] - 1) + lo[inst]
        for _ in range(case["steps"]):
            M = _exact_step(M[:, src], 1, w.K, w.nu, [i], [n[inst]], False, [1], lo[inst])
        return M.float() if case["precision"] == "fp32" else M
    D, shape, pad, a = _flow_args(case)
    if math.prod(shape) * a["RT_hi"] > (9e6 if D == 2 else 1e5):  # over about twenty seconds
        return None
    M = _flow_interior(shape, seed, **a).contiguous()
    full = [n + 2 * pad for n in shape]
    grid = torch.meshgrid(*[torch.arange(-pad, n + pad, device="cuda") for n in shape], indexing="ij")
    index = [v.reshape(-1) for v in reversed(grid)]
    extent = list(reversed(shape))
    stride = [1, full[-1]] + ([full[-1] * full[-2]] if D == 3 else [])
    origin = pad * sum(stride)
    src = sum(v.clamp(min=0).clamp(max=n - 1) * st for v, n, st in zip(index, extent, stride)) + origin
    M = _padded(M, pad).reshape(N_MOM[D], -1)
    for _ in range(case["steps"]):
        M = _exact_step(M[:, src], D, W.internal_dof(GAMMA, D), 1e-3, index, extent, a["periodic"], stride, origin)
    M = M.reshape(N_MOM[D], *full)
    return M.float() if case["precision"] == "fp32" else M
