"""Workloads of the D3V15 solver that its users run, for timing the library.

Every case goes through the package's public calls.  Kinds:

  solve    one run: initial fields -> f = f^eq -> `steps` time steps -> the
           state f (double storage: the fields rho, u, T as well).  `host`
           runs start from numpy arrays and end in numpy arrays, as in the
           package's quick start; the others keep everything on the device.
  batch    several grids advanced together by step_batch, as the batched run
           and the solve server do.
  moments  rho, u, T of a state on the device (end of every served solve).
  conserved  the global mass, momentum and energy sums of a state.
  growth   the von Neumann parameter search of one solve request: max |omega|
           of every candidate (c1, dt) over the request's states.

Flows (`flow`), all of the paper's Sec. 4:
  tube     a Riemann problem along x, x faces held, y and z periodic
  shock    a planar shock entering at x = 0 into gas holding a sphere of
           another density: x-lo held, x-hi extrapolated, y and z periodic
  bubble   the paper's 3D run: the shock comes from x-hi, x-lo extrapolated,
           y and z faces reflect
Initial fields carry a few smooth seeded modes of 2 % on top of the flow.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1010_4135_gb300 import sim as S
from paper_1010_4135_gb300 import stability

NV = 15
GAMMA = 1.4
PERIODIC, FIXED, EXTRAPOLATE, REFLECT = 0, 1, 2, 3


def listed():
    return [
        # the Lax shock tube (Sec. 4(1)) as the quick start runs it: double precision, numpy in and out
        dict(name="lax_tube_fp64", kind="solve", flow="tube", prec="fp64", host=True, nx=200, ny=4, nz=4,
             left_rho=0.445, left_u=0.698, left_p=3.528, right_rho=0.5, right_p=0.571, c1=2.0, eta0=2.0, steps=200),
        # the high-Mach tube (pressure ratio 500) in single precision: 2000 x 4 x 4, thousands of small steps
        dict(name="high_mach_tube_fp32", kind="solve", flow="tube", prec="fp32", host=False, nx=2000, ny=4, nz=4,
             left_rho=5.0, left_u=0.0, left_p=500.0, right_rho=1.0, right_p=1.0, c1=12.0, eta0=20.0, steps=200),
        # the smallest served request: 64^3, alone on the GPU
        dict(name="served_64_fp32", kind="solve", flow="shock", prec="fp32", host=False, nx=64, ny=64, nz=64,
             mach=2.0, sphere=0.5, c1=2.0, eta0=4.0, steps=100),
        # a served grid of middle size
        dict(name="served_128_fp32", kind="solve", flow="shock", prec="fp32", host=False, nx=128, ny=128, nz=128,
             mach=3.0, sphere=0.1, c1=4.0, eta0=8.0, steps=150),
        # the paper's 3D run at its printed size, reflecting walls, x extent not a multiple of any tile
        dict(name="paper_bubble_fp32", kind="solve", flow="bubble", prec="fp32", host=False, nx=300, ny=80, nz=80,
             mach=2.0, sphere=0.1358, c1=2.0, eta0=4.0, steps=100),
        # the benchmark grid: Mach-2 shock into a heavy droplet, 256^3
        dict(name="droplet_256_fp32", kind="solve", flow="shock", prec="fp32", host=False, nx=256, ny=256, nz=256,
             mach=2.0, sphere=5.0, c1=2.0, eta0=4.0, steps=150),
        # residents of the solve server advancing together: four grids of the serving mix
        dict(name="served_batch_fp32", kind="batch", grids="64x64x64,96x96x96,128x128x128,192x128x128",
             mach=3.0, sphere=0.1, c1=4.0, eta0=8.0, steps=100),
        # the largest: 512 x 256 x 256 with eight 128^3 grids in one launch per step
        dict(name="bubbles_batch_fp32", kind="batch", grids="512x256x256" + ",128x128x128" * 8,
             mach=3.0, sphere=0.1, c1=4.0, eta0=8.0, steps=60),
        # the paper's 3D run in double precision (the accuracy reference of the FP32 runs)
        dict(name="paper_bubble_fp64", kind="solve", flow="bubble", prec="fp64", host=False, nx=300, ny=80, nz=80,
             mach=2.0, sphere=4.1538, c1=2.0, eta0=4.0, steps=20),
        # fields of the benchmark grid after a run
        dict(name="moments_256_fp32", kind="moments", prec="fp32", nx=256, ny=256, nz=256),
        # conservation monitor of the benchmark grid
        dict(name="conserved_256_fp32", kind="conserved", prec="fp32", nx=256, ny=256, nz=256),
        # parameter search of one served request (Mach 5 shock, gas of a tenth of the density, 128 cells across)
        dict(name="growth_request", kind="growth", mach=5.0, ratio=0.1, ny=128),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _extents(rng, cells):
    """A box of about `cells` cells with aspect ratios up to about 3, no axis a multiple of anything."""
    ax, ay = _log_uniform(rng, 1.0, 3.0), _log_uniform(rng, 0.7, 1.4)
    side = (cells / (ax * ay)) ** (1.0 / 3.0)
    return max(8, round(side * ax)), max(8, round(side * ay)), max(8, round(side))


def draw(rng):
    kind = rng.choice(["tube", "tube", "shock", "shock", "shock", "bubble", "bubble", "batch", "moments", "conserved",
                       "growth"])
    if kind == "tube":
        prec = rng.choice(["fp64", "fp32"])
        return dict(kind="solve", flow="tube", prec=prec, host=rng.random() < 0.3, nx=round(_log_uniform(rng, 150, 4000)),
                    ny=rng.choice([1, 3, 4, 4, 5]), nz=rng.choice([1, 3, 4, 4, 5]),
                    left_rho=round(rng.uniform(0.4, 2.0), 3), left_u=round(rng.uniform(0.0, 0.7), 3),
                    left_p=round(rng.uniform(1.5, 4.0), 3), right_rho=round(rng.uniform(0.4, 1.0), 3),
                    right_p=round(rng.uniform(0.5, 1.0), 3), c1=2.0, eta0=rng.choice([2.0, 4.0]),
                    steps=rng.randint(50, 200))
    if kind in ("shock", "bubble"):
        prec = rng.choice(["fp64", "fp32", "fp32"])
        if prec == "fp32":
            cells = _log_uniform(rng, 60e3, 16e6)
            steps = max(10, min(200, round(_log_uniform(rng, 4e8, 2.4e9) / cells)))
        else:
            cells = _log_uniform(rng, 30e3, 4e6)
            steps = max(4, min(40, round(_log_uniform(rng, 1e7, 3e7) / cells)))
        nx, ny, nz = _extents(rng, cells)
        return dict(kind="solve", flow=kind, prec=prec, host=False, nx=nx, ny=ny, nz=nz,
                    mach=round(rng.uniform(1.5, 2.5), 2), sphere=round(_log_uniform(rng, 0.2, 4.0), 3), c1=2.0,
                    eta0=4.0, steps=steps)
    if kind == "batch":
        n = rng.randint(2, 8)
        sizes = []
        for _ in range(n):
            if rng.random() < 0.5:
                sizes.append(rng.choice(["64x64x64", "96x96x96", "128x128x128", "192x128x128"]))
            else:
                sizes.append("x".join(str(v) for v in _extents(rng, _log_uniform(rng, 60e3, 4e6))))
        return dict(kind="batch", grids=",".join(sizes), mach=round(rng.uniform(1.5, 3.0), 2),
                    sphere=round(_log_uniform(rng, 0.1, 1.0), 3), c1=4.0, eta0=8.0, steps=rng.randint(20, 100))
    if kind in ("moments", "conserved"):
        nx, ny, nz = _extents(rng, _log_uniform(rng, 200e3, 16e6))
        return dict(kind=kind, prec=rng.choice(["fp64", "fp32", "fp32"]), nx=nx, ny=ny, nz=nz)
    return dict(kind="growth", mach=round(rng.uniform(1.2, 9.0), 2), ratio=round(_log_uniform(rng, 0.1, 10.0), 3),
                ny=rng.choice([64, 96, 128, 256]))


# ---------------------------------------------------------------- inputs

def _shock(mach):
    """(rho, u, p) behind a normal shock of this Mach number moving in +x into (1, 0, 1)."""
    m2 = mach * mach
    rho = (GAMMA + 1.0) * m2 / ((GAMMA - 1.0) * m2 + 2.0)
    p = 1.0 + 2.0 * GAMMA / (GAMMA + 1.0) * (m2 - 1.0)
    return rho, mach * math.sqrt(GAMMA) * (1.0 - 1.0 / rho), p


def _setup(case):
    """Grid, constants and boundary kinds of one solve (the arguments of Sim)."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    flow = case["flow"]
    dx = 1.0 / nx if flow == "tube" else 1.0 / ny
    c1, eta0 = case["c1"], case["eta0"]
    c2 = 3.0 * c1
    dt = 0.04 * dx * math.sqrt(3.0) / c2  # Courant number of the diagonal velocities, as in the paper's runs
    zero = (0.0,) * 5
    if flow == "tube":
        left = (case["left_rho"], case["left_u"], 0.0, 0.0, case["left_p"] / case["left_rho"])
        right = (case["right_rho"], 0.0, 0.0, 0.0, case["right_p"] / case["right_rho"])
        lo, hi = (FIXED, PERIODIC, PERIODIC), (FIXED, PERIODIC, PERIODIC)
        fixed_lo, fixed_hi = (left, zero, zero), (right, zero, zero)
    else:
        rho, u, p = _shock(case["mach"])
        if flow == "shock":
            lo, hi = (FIXED, PERIODIC, PERIODIC), (EXTRAPOLATE, PERIODIC, PERIODIC)
            fixed_lo, fixed_hi = ((rho, u, 0.0, 0.0, p / rho), zero, zero), (zero, zero, zero)
        else:
            lo, hi = (EXTRAPOLATE, REFLECT, REFLECT), (FIXED, REFLECT, REFLECT)
            fixed_lo, fixed_hi = (zero, zero, zero), ((rho, -u, 0.0, 0.0, p / rho), zero, zero)
    return dict(nx=nx, ny=ny, nz=nz, c1=c1, c2=c2, eta0=eta0, tau=dt, dt=dt, dx=dx, gamma=GAMMA,
                bc_lo=lo, bc_hi=hi, fixed_lo=fixed_lo, fixed_hi=fixed_hi)


def _modes(shape, rng):
    """A sum of three seeded products of cosines over the box, at most 1 in size."""
    nz, ny, nx = shape
    out = torch.zeros(shape, dtype=torch.float64, device="cuda")
    for _ in range(3):
        f = []
        for n in (nz, ny, nx):
            x = torch.arange(n, dtype=torch.float64, device="cuda") * (2.0 * math.pi / n)
            f.append(torch.cos(int(rng.integers(0, 4)) * x + float(rng.uniform(0.0, 2.0 * math.pi))))
        out += float(rng.uniform(-1.0, 1.0)) / 3.0 * f[0][:, None, None] * f[1][None, :, None] * f[2][None, None, :]
    return out


def _fields(case, seed, amp=0.02):
    """(rho, u, T) of the flow on the device, double precision, with the seeded modes on top."""
    k = _setup(case)
    nx, ny, nz, dx = k["nx"], k["ny"], k["nz"], k["dx"]
    shape = (nz, ny, nx)

    def centres(n):
        return (torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) * dx

    if case["flow"] == "tube":
        left = (centres(nx) < 0.5)[None, None, :].expand(shape)
        rho = torch.where(left, case["left_rho"], case["right_rho"]).to(torch.float64)
        p = torch.where(left, case["left_p"], case["right_p"]).to(torch.float64)
        ux = torch.where(left, case["left_u"], 0.0).to(torch.float64)
    else:
        lx, lz = nx * dx, nz * dx
        bubble = case["flow"] == "bubble"
        cx, radius = ((2.0 / 3.0) * lx, 0.3 * min(1.0, lz)) if bubble else (0.3 * lx, 0.15 * min(1.0, lz))
        r2 = ((centres(nz) - 0.5 * lz) ** 2)[:, None, None] + ((centres(ny) - 0.5) ** 2)[None, :, None] \
            + ((centres(nx) - cx) ** 2)[None, None, :]
        inside = 0.5 * (1.0 - torch.tanh((r2.sqrt() - radius) / dx))  # a surface one cell thick
        rho = 1.0 + inside * (case["sphere"] - 1.0)
        p = torch.ones(shape, dtype=torch.float64, device="cuda")
        ux = torch.zeros(shape, dtype=torch.float64, device="cuda")
        if bubble:  # the shock stands at five sixths of the length, the shocked gas behind it
            rs, us, ps = _shock(case["mach"])
            behind = (centres(nx) >= (5.0 / 6.0) * lx)[None, None, :].expand(shape)
            rho, p, ux = torch.where(behind, rs, rho), torch.where(behind, ps, p), torch.where(behind, -us, ux)
    T = p / rho
    rng = np.random.default_rng([seed, nx, ny, nz])
    rho = rho * (1.0 + amp * _modes(shape, rng))
    T = T * (1.0 + amp * _modes(shape, rng))
    u = torch.stack([ux + amp * _modes(shape, rng), amp * _modes(shape, rng), amp * _modes(shape, rng)])
    return rho.contiguous(), u, T.contiguous()


def _grids(case):
    """The solves of a batch, one per grid of its list."""
    out = []
    for g in case["grids"].split(","):
        nx, ny, nz = (int(v) for v in g.split("x"))
        out.append(dict(case, kind="solve", flow="shock", prec="fp32", nx=nx, ny=ny, nz=nz))
    return out


# a state to be measured: a smooth flow with 2 % seeded noise on the populations
_STATE = dict(flow="shock", mach=2.0, sphere=5.0, c1=2.0, eta0=4.0)


def _state_f(case, seed):
    k = _setup(dict(case, **_STATE))
    f = _feq(k, *_fields(dict(case, **_STATE), seed))
    g = torch.Generator(device="cuda").manual_seed(seed)
    f *= 1.0 + 0.02 * (2.0 * torch.rand(f.shape, generator=g, device="cuda", dtype=torch.float64) - 1.0)
    return f if case["prec"] == "fp64" else f.to(torch.float32)


def _request(case, seed):
    """States and candidate parameter sets of one solve request (the seed varies its states by up to 2 %)."""
    rng = np.random.default_rng(seed)

    def vary(x):
        return x * (1.0 + 0.02 * float(rng.uniform(-1.0, 1.0)))

    rho, u, p = _shock(case["mach"])
    ratio = case["ratio"]
    pre, post, other = (1.0, 0.0, 0.0, 0.0, 1.0), (rho, u, 0.0, 0.0, p / rho), (ratio, 0.0, 0.0, 0.0, 1.0 / ratio)
    # two states between the shocked gas and the second gas, as where the shock has crossed the interface
    mid = tuple((a + 2.0 * b) / 3.0 for a, b in zip(post, other))
    fast = (0.5 * rho, 1.2 * u, 0.0, 0.0, 1.5 * p / rho)
    states = [tuple(vary(x) for x in s) for s in (pre, post, other, mid, fast)]
    umax = 1.2 * u
    params = []
    for c1 in sorted({float(max(2, math.ceil(f * umax))) for f in (1.0, 1.1, 1.2, 1.35, 1.5)}):
        for dt in (5e-5, 2e-5, 1e-5, 5e-6, 2e-6, 1e-6, 5e-7, 2e-7):
            if 3.0 * c1 / math.sqrt(3.0) * dt * case["ny"] <= 0.025:
                params.append((c1, 3.0 * c1, 2.0 * c1, GAMMA, dt, dt, 1.0 / case["ny"]))
    return states, params


def prepare(case, seed):
    kind = case["kind"]
    if kind == "growth":
        states, params = _request(case, seed)
        return dict(kind=kind, states=states, params=params)
    if kind in ("moments", "conserved"):
        k = _setup(dict(case, **_STATE))
        s = S.Sim(precision=case["prec"], **k)
        s.set_f(_state_f(case, seed))
        s.sync()
        return dict(kind=kind, sim=s)
    solves = _grids(case) if kind == "batch" else [case]
    sims, fields, outs = [], [], []
    for i, c in enumerate(solves):
        s = S.Sim(precision=c["prec"], **_setup(c))
        rho, u, T = _fields(c, seed + 1000 * i)
        if c.get("host"):
            fields.append(tuple(x.cpu().numpy() for x in (rho, u, T)))
            outs.append(None)
        else:
            fields.append((rho, u, T))
            outs.append(torch.empty((NV,) + s.shape, device="cuda",
                                    dtype=torch.float64 if c["prec"] == "fp64" else torch.float32))
        sims.append(s)
    return dict(kind=kind, sims=sims, fields=fields, outs=outs, steps=case["steps"], host=bool(case.get("host")),
                prec=solves[0]["prec"])


# ---------------------------------------------------------------- one pass

def run(state):
    kind = state["kind"]
    if kind == "growth":
        return stability.max_growth_device(state["states"], state["params"], nk=24)
    if kind == "moments":
        return state["sim"].moments(on_device=True)
    if kind == "conserved":
        return state["sim"].conserved()
    for s, (rho, u, T) in zip(state["sims"], state["fields"]):
        s.init(rho, u, T)
    if kind == "batch":
        S.step_batch(state["sims"], state["steps"])
    else:
        state["sims"][0].step(state["steps"])
    if state["host"]:
        s = state["sims"][0]
        return (s.get_f(),) + (s.moments() if state["prec"] == "fp64" else ())
    out = [s.get_f(out=f) for s, f in zip(state["sims"], state["outs"])]
    if kind == "solve" and state["prec"] == "fp64":
        out += list(state["sims"][0].moments(on_device=True))
    return out


def work(case):
    """Bytes: every step reads and writes the 15 populations once; the initial fields are read and the results
    written once.  Operations: per cell and step about 50 for the moments, 70 for the equilibrium, 270 for the 30
    limited gradients, 55 for the dissipation term and 75 for the update."""
    kind = case["kind"]
    if kind == "growth":
        states, params = _request(case, 0)
        n = len(states) * len(params) * 2 * 24
        # per matrix: Hessenberg reduction (10/3 n^3) and QR eigenvalues (about 7 n^3), complex (4 fused each)
        return {"bytes": 8.0 * (7 * len(params) + 5 * len(states)), "flops": n * 2.0 * 4.0 * (10.0 / 3.0 + 7.0) * NV ** 3}
    if kind == "batch":
        w = [work(c) for c in _grids(case)]
        return {k: sum(x[k] for x in w) for k in ("bytes", "flops")}
    cells = float(case["nx"] * case["ny"] * case["nz"])
    size = 8 if case["prec"] == "fp64" else 4
    if kind == "moments":
        return {"bytes": cells * (NV * size + 5 * 8), "flops": cells * 55}
    if kind == "conserved":
        return {"bytes": cells * NV * size, "flops": cells * 30}
    out = NV * size + (5 * 8 if case["prec"] == "fp64" else 0)
    return {"bytes": cells * (case["steps"] * 2 * NV * size + 5 * 8 + out),
            "flops": cells * (case["steps"] * 520.0 + 120.0)}


# ---------------------------------------------------------------- the same in 64 bits, plainly

def _velocities(k):
    s = k["c2"] / math.sqrt(3.0)
    v = [[0.0, 0.0, 0.0]]
    for a in range(3):
        for sign in (1.0, -1.0):
            v.append([sign * k["c1"] if b == a else 0.0 for b in range(3)])
    for sx in (1.0, -1.0):
        for sy in (1.0, -1.0):
            for sz in (1.0, -1.0):
                v.append([s * sx, s * sy, s * sz])
    return v


def _feq(k, rho, u, T):
    """f^eq of the paper (Sec. 2): rho (A_i + B_i v.u + D_i (v.u)^2)."""
    c1, c2, eta0 = k["c1"], k["c2"], k["eta0"]
    b = 2.0 / (k["gamma"] - 1.0)
    u2 = u[0] * u[0] + u[1] * u[1] + u[2] * u[2]
    f = torch.empty((NV,) + tuple(rho.shape), dtype=torch.float64, device=rho.device)
    for i, v in enumerate(_velocities(k)):
        if i == 0:
            f[0] = rho * ((b - 3.0) / eta0 ** 2) * T
            continue
        if i <= 6:
            A = (-c2 ** 2 + ((b - 3.0) * c2 ** 2 / eta0 ** 2 + 3.0) * T + (c2 / c1) ** 2 * u2) / (6.0 * (c1 ** 2 - c2 ** 2))
            B = (-c2 ** 2 + (b + 2.0) * T + u2) / (2.0 * c1 ** 2 * (c1 ** 2 - c2 ** 2))
            D = 1.0 / (2.0 * c1 ** 4)
        else:
            A = (-c1 ** 2 + ((b - 3.0) * c1 ** 2 / eta0 ** 2 + 3.0) * T + (3.0 * c1 ** 2 - c2 ** 2) / (2.0 * c2 ** 2) * u2) \
                / (8.0 * (c2 ** 2 - c1 ** 2))
            B = 3.0 * (-c1 ** 2 + (b + 2.0) * T + u2) / (8.0 * c2 ** 2 * (c2 ** 2 - c1 ** 2))
            D = 9.0 / (16.0 * c2 ** 4)
        w = v[0] * u[0] + v[1] * u[1] + v[2] * u[2]
        f[i] = rho * (A + B * w + D * w * w)
    return f


def _macros(k, f):
    """(rho, u, T) of populations f [15, ...]."""
    v = _velocities(k)
    b = 2.0 / (k["gamma"] - 1.0)
    rho, mom, energy = torch.zeros_like(f[0]), [torch.zeros_like(f[0]) for _ in range(3)], torch.zeros_like(f[0])
    for i in range(NV):
        rho += f[i]
        for a in range(3):
            if v[i][a]:
                mom[a] += v[i][a] * f[i]
        energy += (sum(c * c for c in v[i]) + (k["eta0"] ** 2 if i == 0 else 0.0)) * f[i]
    u = torch.stack([m / rho for m in mom])
    return rho, u, (energy / rho - (u[0] * u[0] + u[1] * u[1] + u[2] * u[2])) / b


def _ghosts(k, g):
    """The two layers outside each face of the padded populations g [15, nz+4, ny+4, nx+4] (Sec. 4(2))."""
    for axis in range(3):
        dim = 3 - axis
        n = g.shape[dim] - 4
        inner = [slice(None)] + [slice(2, -2)] * 3

        def at(j):
            s = list(inner)
            s[dim] = j + 2
            return tuple(s)

        for side, kind, fixed in ((0, k["bc_lo"][axis], k["fixed_lo"][axis]), (1, k["bc_hi"][axis], k["fixed_hi"][axis])):
            near, far = (-1, -2) if side == 0 else (n, n + 1)
            if kind == PERIODIC:
                g[at(near)], g[at(far)] = g[at(near % n)].clone(), g[at(far % n)].clone()
                continue
            m0 = _macros(k, g[at(0 if side == 0 else n - 1)])
            if kind == FIXED:
                one = torch.ones_like(m0[0])
                m1 = (fixed[0] * one, torch.stack([fixed[1 + a] * one for a in range(3)]), fixed[4] * one)
                m2 = m1
            elif kind == EXTRAPOLATE:
                m_in = _macros(k, g[at(1 if side == 0 else n - 2)])
                m1 = tuple(2.0 * a - c for a, c in zip(m0, m_in))
                m2 = tuple(2.0 * a - c for a, c in zip(m1, m0))
            else:
                u1, u2 = m0[1].clone(), m0[1].clone()
                u1[axis] = 0.0
                u2[axis] = -u2[axis]
                m1, m2 = (m0[0], u1, m0[2]), (m0[0], u2, m0[2])
            g[at(near)], g[at(far)] = _feq(k, *m1), _feq(k, *m2)


def _minmod(a, b):
    return torch.where(a * b > 0.0, torch.where(a.abs() < b.abs(), a, b), 0.0)


def _advance(k, f, steps):
    """`steps` time steps (Sec. 3: NND convection, the dissipation term, relaxation, forward Euler) of f [15, nz, ny, nx]."""
    nz, ny, nx = f.shape[1:]
    g = torch.zeros((NV, nz + 4, ny + 4, nx + 4), dtype=torch.float64, device=f.device)
    inner = (slice(None),) + (slice(2, -2),) * 3
    g[inner] = f
    v = _velocities(k)
    dt, dx, tau = k["dt"], k["dx"], k["tau"]
    for _ in range(steps):
        _ghosts(k, g)
        new = _feq(k, *_macros(k, g[inner]))
        for i in range(NV):
            q = g[i]

            def near(dim, d):
                s = [slice(2, -2)] * 3
                s[dim] = slice(2 + d, q.shape[dim] - 2 + d)
                return q[tuple(s)]

            c = near(0, 0)
            rate = (new[i] - c) / tau
            lam = k["c1"] * dx if i == 0 else (0.1 * k["c1"] * dx if i <= 6 else 0.0)
            for a in range(3):
                d, va = 2 - a, v[i][a]
                m1, p1 = near(d, -1), near(d, 1)
                if va > 0.0:
                    e = c - m1
                    rate -= va / dx * (e + 0.5 * (_minmod(p1 - c, e) - _minmod(m1 - near(d, -2), e)))
                elif va < 0.0:
                    e = p1 - c
                    rate -= va / dx * (e - 0.5 * (_minmod(near(d, 2) - p1, e) - _minmod(c - m1, e)))
                if lam:
                    rate += lam / dx ** 2 * ((p1 - c) - (c - m1))
            new[i] = c + dt * rate
        g[inner] = new
    return g[inner].contiguous()


def exact(case, seed):
    kind = case["kind"]
    if kind == "growth":
        states, params = _request(case, seed)
        return _growth(states, params, 24)
    if kind in ("moments", "conserved"):
        k = _setup(dict(case, **_STATE))
        f = _state_f(case, seed).to(torch.float64)
        if kind == "moments":
            return _macros(k, f)
        v = _velocities(k)
        total = [f[i].sum().item() for i in range(NV)]
        e = [sum(c * c for c in v[i]) + (k["eta0"] ** 2 if i == 0 else 0.0) for i in range(NV)]
        return np.array([math.fsum(total)] + [math.fsum(v[i][a] * total[i] for i in range(NV)) for a in range(3)]
                        + [math.fsum(e[i] * total[i] for i in range(NV))])
    out = []
    for i, c in enumerate(_grids(case) if kind == "batch" else [case]):
        k = _setup(c)
        f = _feq(k, *_fields(c, seed + 1000 * i))
        if c["prec"] == "fp32":
            f = f.to(torch.float32).to(torch.float64)
        f = _advance(k, f, case["steps"])
        out.append(f)
        if c["prec"] == "fp64":
            out += list(_macros(k, f))
    return out


def _growth(states, params, nk):
    """max |omega| of the amplification matrix G (Sec. 3, first-order upwind phases) of each parameter set."""
    worst = np.zeros(len(params))
    for p, (c1, c2, eta0, gamma, dt, tau, dx) in enumerate(params):
        k = dict(c1=c1, c2=c2, eta0=eta0, gamma=gamma)
        v = np.array(_velocities(k))
        eta2 = np.zeros(NV)
        eta2[0] = eta0 ** 2
        b = 2.0 / (gamma - 1.0)
        lam = np.array([c1 * dx] + [0.1 * c1 * dx] * 6 + [0.0] * 8)
        for rho, u1, u2, u3, T in states:
            u = np.array([u1, u2, u3])
            rel = v - u
            # columns: d(rho, u, T)/df_j; rows: df^eq_i/d(rho, u, T)
            dm = np.vstack([np.ones(NV), (rel / rho).T, ((rel * rel).sum(1) + eta2 - b * T) / (b * rho)])
            J = _feq_gradient(k, rho, u, T) @ dm
            for d in ((1.0, 0.0, 0.0), (1.0, 1.0, 1.0)):
                d = np.array(d) / np.linalg.norm(d)
                th = (np.pi / nk * np.arange(1, nk + 1))[:, None] * d[None, :]
                plus, minus = 1.0 - np.exp(-1j * th), np.exp(1j * th) - 1.0
                phi = np.where(v[None] >= 0.0, plus[:, None, :], minus[:, None, :])
                diag = 1.0 - dt / tau - (v[None] * phi).sum(2) * dt / dx \
                    + lam[None] * dt / dx ** 2 * (2.0 * np.cos(th) - 2.0).sum(1)[:, None]
                G = dt / tau * np.broadcast_to(J, (nk, NV, NV)).astype(complex)
                G = G + diag[:, :, None] * np.eye(NV)
                worst[p] = max(worst[p], np.abs(np.linalg.eigvals(G)).max())
    return worst


def _feq_gradient(k, rho, u, T):
    """df^eq_i/d(rho, u1, u2, u3, T) [15, 5]: f^eq is rho times a polynomial of the second degree in u and T, so
    automatic differentiation of it is exact."""
    x = torch.tensor([rho, *u, T], dtype=torch.float64)
    return torch.autograd.functional.jacobian(lambda y: _feq_vector(k, y), x).numpy()


def _feq_vector(k, y):
    c1, c2, eta0 = k["c1"], k["c2"], k["eta0"]
    b = 2.0 / (k["gamma"] - 1.0)
    rho, u, T = y[0], y[1:4], y[4]
    u2 = (u * u).sum()
    w = torch.tensor(_velocities(k), dtype=torch.float64) @ u
    Aa = (-c2 ** 2 + ((b - 3.0) * c2 ** 2 / eta0 ** 2 + 3.0) * T + (c2 / c1) ** 2 * u2) / (6.0 * (c1 ** 2 - c2 ** 2))
    Ba = (-c2 ** 2 + (b + 2.0) * T + u2) / (2.0 * c1 ** 2 * (c1 ** 2 - c2 ** 2))
    Ad = (-c1 ** 2 + ((b - 3.0) * c1 ** 2 / eta0 ** 2 + 3.0) * T + (3.0 * c1 ** 2 - c2 ** 2) / (2.0 * c2 ** 2) * u2) \
        / (8.0 * (c2 ** 2 - c1 ** 2))
    Bd = 3.0 * (-c1 ** 2 + (b + 2.0) * T + u2) / (8.0 * c2 ** 2 * (c2 ** 2 - c1 ** 2))
    axis = rho * (Aa + Ba * w[1:7] + w[1:7] ** 2 / (2.0 * c1 ** 4))
    diagonal = rho * (Ad + Bd * w[7:] + w[7:] ** 2 * 9.0 / (16.0 * c2 ** 4))
    return torch.cat([(rho * ((b - 3.0) / eta0 ** 2) * T).reshape(1), axis, diagonal])
