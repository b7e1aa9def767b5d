"""The work a user of this library has it do, as measurable cases.

A pass is what a solve is: the initial level goes into an existing solver (device tensors), the
solver advances `steps` time levels, and the new level comes out as device tensors.  The solver
(its level buffers, maps and coefficients) is what a program keeps between solves.

Families, all on periodic grids, with the parameters of `paper_2505_17057_gb300/configs.py` and
`serving.py`:

  cde2d     linear CDE, D2Q9, two levels (cde2d_64, lcde2d_8192)
  ncde2d    nonlinear CDE, D2Q9, three levels (ncde2d_1024, the serving stream)
  nse2d     He-Luo NSE, D2Q9, two levels (tgv2d_4096); viscosity 1/6 (LBGK tau = 1) or less
  cde3d     linear CDE, D3Q7, two levels (cde3d_512)
  ncde3d    nonlinear CDE, D3Q19, three levels (the serving stream)
  nse3d     He-Luo NSE, D3Q19, two levels (nse3d_512)
  srccde2d  linear CDE with a time-dependent source set before every step, three levels
            (srccde2d_4096)
  theta2d   Crank-Nicolson steps of the linear CDE at dt = 8 (theta2d_4096)

Fields enter and leave in FP32 (FP32 / BF16 storage) or FP64 (FP64 storage).
"""
from __future__ import annotations

import math
import random

import torch

from paper_2505_17057_gb300 import mmfd

THREE_A = (7 / 8, 0.0, 1 / 8)
THREE_AHAT = (1 / 8, 0.0, -1 / 8)
K2 = [[0.02, 0.005], [0.005, 0.01]]
U2 = [0.1, 0.05]
K3 = (0.02, 0.015, 0.01)
U3 = (0.05, 0.03, 0.02)
THETA_DT = 8.0
DIM3 = ("cde3d", "ncde3d", "nse3d")


def _case(name, family, n, steps, storage="fp32", depth=1, a0=0.0, sr=False):
    c = {"family": family, "nx": n[0], "ny": n[1], "nz": n[2] if len(n) > 2 else 1, "steps": steps,
         "storage": storage, "depth": depth, "a0": a0, "sr": sr}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest grid of the configurations, in the accuracy tier's storage: a step is a few
        # microseconds of launch and latency
        _case("cde2d_64_fp64", "cde2d", (64, 64), 200, storage="fp64"),
        # a small flow solve of the size a parameter study or a served request has, odd-sized, at a
        # viscosity other than the LBGK tau = 1 one
        _case("nse2d_250x181", "nse2d", (250, 181), 200, a0=0.5),
        # the nonlinear CDE configuration: three levels that stay in L2
        _case("ncde2d_1024", "ncde2d", (1024, 1024), 100),
        # the scalar bandwidth probe at the default one step per launch
        _case("lcde2d_8192", "cde2d", (8192, 8192), 48),
        # the headline workload: Taylor-Green at 4096^2, steps per launch left to the library
        _case("tgv2d_4096", "nse2d", (4096, 4096), 60, depth=0),
        # a large ragged flow grid in the low-memory tier with stochastic rounding, as served
        _case("tgv2d_3001x2047_bf16", "nse2d", (3001, 2047), 40, storage="bf16", sr=True),
        # the accuracy reference run of the flow solver
        _case("tgv2d_1000x800_fp64", "nse2d", (1000, 800), 10, storage="fp64"),
        # the 3D linear CDE configuration
        _case("cde3d_512", "cde3d", (512, 512, 512), 24),
        # the 3D flow configuration (the heaviest per node)
        _case("nse3d_512", "nse3d", (512, 512, 512), 20),
        # a 3D nonlinear request of the serving stream's range, narrower than a marching strip
        _case("ncde3d_96", "ncde3d", (96, 96, 96), 40),
        # a time-dependent source, uploaded from the device before every step
        _case("srccde2d_4096", "srccde2d", (4096, 4096), 10),
        # implicit steps: a right-hand side and Jacobi sweeps per step
        _case("theta2d_4096", "theta2d", (4096, 4096), 8, depth=0),
    ]


def draw(rng):
    """One more case of the listed ranges: sizes log-uniform (and mostly not round), sides of a grid
    within a factor of two of each other, steps so that a pass costs no more than the largest
    listed one."""
    family = rng.choice(["cde2d", "cde2d", "nse2d", "nse2d", "nse2d", "ncde2d", "cde3d", "nse3d", "nse3d", "ncde3d",
                         "srccde2d", "theta2d"])
    storage = "fp32"
    if family not in ("srccde2d", "theta2d"):
        storage = rng.choices(["fp32", "bf16", "fp64"], [6, 2, 2])[0]
    if family in DIM3:
        top = 512 if storage != "fp64" else 144
        side = math.exp(rng.uniform(math.log(32), math.log(top / 1.25)))
        n = tuple(min(top, max(16, int(side * rng.uniform(0.8, 1.25)))) for _ in range(3))
    else:
        top = {"cde2d": 8192, "nse2d": 4096, "ncde2d": 2048, "srccde2d": 4096, "theta2d": 4096}[family]
        if storage == "fp64":
            top = 2048
        low = 128 if family == "theta2d" else 32
        side = math.exp(rng.uniform(math.log(low), math.log(top / 1.4)))
        n = tuple(min(top, max(low, int(side * rng.uniform(0.7, 1.4)))) for _ in range(2))
    # about 3e8 node updates, 4 to 200 steps; FP64 and the heavier node updates take fewer
    weight = {"cde2d": 1, "ncde2d": 4, "nse2d": 4, "cde3d": 1, "ncde3d": 8, "nse3d": 8, "srccde2d": 2, "theta2d": 10}
    per = math.prod(n) * weight[family] * (40 if storage == "fp64" else 1)
    steps = max(4, min(200, int(3e8 / per) if family not in ("srccde2d", "theta2d") else min(10, int(3e8 / per))))
    depth = 1
    a0 = 0.0
    if family == "theta2d":
        depth = 0
    elif family in ("cde2d", "nse2d"):
        depth = rng.choice([0, 1])
    if family in ("nse2d", "nse3d"):
        a0 = rng.choice([0.0, 0.0, 0.5])
    # round-to-nearest stalls the slow scalar problems in BF16: those use stochastic rounding
    sr = storage == "bf16" and (family not in ("nse2d", "nse3d") or rng.random() < 0.7)
    return _case(None, family, n, steps, storage=storage, depth=depth, a0=a0, sr=sr)


# ------------------------------------------------------------------ inputs

def _modes2d(rnd, nx, ny, count, lo, hi, kmax):
    """sum_m A_m cos(k_m . x + t_m) on the periodic box, as one matrix product."""
    x = 2 * math.pi * torch.arange(nx, dtype=torch.float64, device="cuda") / nx
    y = 2 * math.pi * torch.arange(ny, dtype=torch.float64, device="cuda") / ny
    cols, rows = [], []
    for _ in range(count):
        a, t = rnd.uniform(lo, hi), rnd.uniform(0, 2 * math.pi)
        kx, ky = rnd.randint(1, kmax), rnd.randint(-kmax, kmax)
        cols += [torch.cos(ky * y), -torch.sin(ky * y)]
        rows += [a * torch.cos(kx * x + t), a * torch.sin(kx * x + t)]
    return torch.stack(cols, 1) @ torch.stack(rows, 0)


def _series(rnd, n, nmodes):
    """A random cosine series of the periodic axis with max |S| = 1, and its derivative."""
    x = 2 * math.pi * torch.arange(n, dtype=torch.float64, device="cuda") / n
    s, d = torch.zeros_like(x), torch.zeros_like(x)
    for m in range(1, nmodes + 1):
        a, t = rnd.uniform(0.1, 0.5), rnd.uniform(0, 2 * math.pi)
        s += a * torch.cos(m * x + t)
        d -= a * m * torch.sin(m * x + t)
    top = s.abs().max()
    return s / top, d / top


def _inputs(case, seed):
    """The initial level in the case's field type: [fields of level t], [fields of t - dt or None],
    sources per step or None."""
    rnd = random.Random(seed)
    dt = torch.float64 if case["storage"] == "fp64" else torch.float32
    nx, ny, nz, fam = case["nx"], case["ny"], case["nz"], case["family"]
    prev = src = None
    if fam in ("cde2d", "theta2d"):
        if nx * ny <= 128 * 128:
            x = torch.arange(nx, dtype=torch.float64, device="cuda")[None, :]
            y = torch.arange(ny, dtype=torch.float64, device="cuda")[:, None]
            cx, cy = nx / 2 + rnd.uniform(-2, 2), ny / 2 + rnd.uniform(-2, 2)
            f = [torch.exp(-((x - cx) ** 2 + (y - cy) ** 2) / (2.0 * rnd.uniform(5, 7) ** 2))]
        else:
            f = [1.0 + _modes2d(rnd, nx, ny, 32, 0.1, 0.5, 8)]
    elif fam == "ncde2d":
        p = _modes2d(rnd, nx, ny, 32, 0.1, 0.5, 6)
        f = [p * (NCDE_TOP / p.abs().max())]
    elif fam == "ncde3d":
        p = _outer(_series(rnd, nx, 4)[0], _series(rnd, ny, 4)[0], _series(rnd, nz, 4)[0])
        f = [NCDE_TOP * p]
    elif fam == "cde3d":
        f = [1.0 + 0.5 * _outer(_series(rnd, nx, 16)[0], _series(rnd, ny, 16)[0], _series(rnd, nz, 16)[0])]
    elif fam == "nse2d":
        u0 = min(100 * (1 / 6) / min(nx, ny), 0.05)
        kx, ky = 2 * math.pi / nx, 2 * math.pi / ny
        x = kx * torch.arange(nx, dtype=torch.float64, device="cuda")[None, :] + rnd.uniform(0, 2 * math.pi)
        y = ky * torch.arange(ny, dtype=torch.float64, device="cuda")[:, None] + rnd.uniform(0, 2 * math.pi)
        u = -u0 * torch.cos(x) * torch.sin(y)
        v = u0 * (kx / ky) * torch.sin(x) * torch.cos(y)
        rho = 1.0 - 0.75 * u0 * u0 * (torch.cos(2 * x) + (kx / ky) ** 2 * torch.cos(2 * y))
        f = [rho, u, v]
    elif fam == "nse3d":
        (P, dP), (R, dR), (U, dU) = _series(rnd, ny, 8), _series(rnd, nx, 8), _series(rnd, nx, 8)
        (Q, dQ), (T, dT), (V, dV) = _series(rnd, nz, 8), _series(rnd, nz, 8), _series(rnd, ny, 8)
        one = [torch.ones(m, dtype=torch.float64, device="cuda") for m in (nx, ny, nz)]
        ux = _outer(U, dV, one[2]) - _outer(R, one[1], dT)
        uy = _outer(one[0], P, dQ) - _outer(dU, V, one[2])
        uz = _outer(dR, one[1], T) - _outer(one[0], dP, Q)
        s = 0.05 / max(float(w.abs().max()) for w in (ux, uy, uz))
        f = [torch.ones_like(ux), ux * s, uy * s, uz * s]
    else:   # srccde2d: Example 1's field and source at a random phase
        d, kappa = _src_scales(case)
        x = d["dx"] * torch.arange(nx, dtype=torch.float64, device="cuda")[None, :]
        y = d["dx"] * torch.arange(ny, dtype=torch.float64, device="cuda")[:, None]
        # whole wave numbers of the box, close to pi on the square one
        kx, ky = 2 * math.pi / (nx * d["dx"]), 2 * math.pi / (ny * d["dx"])
        t = kx * x + ky * y + rnd.uniform(0, 2 * math.pi)
        g = 1.0 - (kx * kx + ky * ky) * kappa
        s, base = torch.sin(t), torch.sin(t) + (0.1 * kx + 0.1 * ky) * torch.cos(t)
        f, prev = [s], [math.exp(-g * d["dt"]) * s]
        src = [[(math.exp(g * m * d["dt"]) * base).to(dt).contiguous()] for m in range(case["steps"])]
    cast = lambda fs: None if fs is None else [w.to(dt).contiguous() for w in fs]
    return cast(f), cast(prev), src


def _outer(sx, sy, sz):
    return sz[:, None, None] * sy[None, :, None] * sx[None, None, :]


# ------------------------------------------------------------------ the problem statements

NCDE_TOP = 2.0   # max |phi0| of the NCDE fields


def _ncde_scales(case):
    """(dx, dt): the diffusive limit of the configuration, a convective one for coarse grids, and
    dt <= 0.5 D_min / max |B'|^2 (as the serving stream chooses its steps)."""
    dx = 2 * math.pi / case["nx"]
    share = 0.4 if case["family"] == "ncde2d" else 0.3
    dmax = 0.01 * (1 + NCDE_TOP ** 2)
    return dx, min(share * dx * dx / (2 * dmax), 0.15 * dx / NCDE_TOP, 0.5 * 0.01 / NCDE_TOP ** 2)


def _src_scales(case):
    half = case["nx"] / 2
    dx = 2.0 / case["nx"]
    dt = 1.0 / (0.06 * half * half)
    return {"dx": dx, "dt": dt}, (dx / dt) ** 2 / 3.0 * dt / 2.0


def _desc(case):
    fam = case["family"]
    dim = 3 if fam in DIM3 else 2
    n = [case["nx"], case["ny"], case["nz"]][:dim]
    kw = dict(n=n, dt=1.0, dx=[1.0] * dim, storage=case["storage"], temporal_depth=case["depth"])
    if case["sr"]:
        kw.update(flags=mmfd.MMFD_FLAG_STOCHASTIC_ROUND, seed=11)
    if fam in ("cde2d", "theta2d"):
        kw.update(pde="LCDE", lattice="D2Q9", levels=2, K=K2, u=U2, targets=[0, -1, -1, 0, 0.5])
        kw["ref"] = [0.0 if n[0] * n[1] <= 128 * 128 else 1.0]
        if fam == "theta2d":
            kw.update(dt=THETA_DT, theta=0.5)
    elif fam == "cde3d":
        kw.update(pde="LCDE", lattice="D3Q7", levels=2, K=[[K3[0], 0, 0], [0, K3[1], 0], [0, 0, K3[2]]], u=U3,
                  targets=[0, -1, -1, 0, 0.5], ref=[1.0])
    elif fam in ("ncde2d", "ncde3d"):
        dx, dt = _ncde_scales(case)
        kw.update(pde="NCDE", lattice="D2Q9" if dim == 2 else "D3Q19", levels=3, dt=dt, dx=[dx] * dim,
                  flux=[[0, 0, 0.5, 0]] * dim, diff=[0.01, 0, 0.01, 0], a=THREE_A, ahat=THREE_AHAT)
    elif fam in ("nse2d", "nse3d"):
        a0 = case["a0"]
        kw.update(pde="NSE", lattice="D2Q9" if dim == 2 else "D3Q19", levels=2, a=(1.0, 0.0, 0.0),
                  abar=(1.0 - a0 / 2, a0, -a0 / 2), ref=[1.0] + [0.0] * dim)
    else:
        d, kappa = _src_scales(case)
        kw.update(pde="LCDE", lattice="D2Q9", levels=3, dt=d["dt"], dx=[d["dx"]] * 2, K=[[kappa, 0], [0, kappa]],
                  u=[0.1, 0.1], a=THREE_A, ahat=THREE_AHAT, source="su", b=(1.5, 0.0, 0.0), bhat=(-0.5, 0.0, 0.0))
    return kw


def prepare(case, seed):
    cur, prev, src = _inputs(case, seed)
    return {"solver": mmfd.Solver(mmfd.make_desc(**_desc(case))), "cur": cur, "prev": prev, "src": src,
            "steps": case["steps"], "dtype": "float64" if case["storage"] == "fp64" else "float32"}


def run(state):
    s = state["solver"]
    s.set_fields(state["cur"])
    if state["prev"] is not None:
        s.set_fields(state["prev"], level=1)
    if state["src"] is not None:
        for q in state["src"]:
            s.set_source(q)
            s.step(1)
    else:
        s.step(state["steps"])
    return s.fields(device=True, dtype=_NP[state["dtype"]])


def _np_types():
    import numpy as np
    return {"float32": np.float32, "float64": np.float64}


_NP = _np_types()


# floating point operations of one node update (multiplies and adds of the collapsed update:
# every direction's contribution formed once per input node, each moment summed once)
FLOPS = {"cde2d": 18, "cde3d": 14, "ncde2d": 136, "ncde3d": 250, "nse2d": 68, "nse3d": 140, "srccde2d": 72,
         "theta2d": 18 + 17 * 20}


def work(case):
    fam = case["family"]
    nodes = case["nx"] * case["ny"] * case["nz"]
    nf = {"nse2d": 3, "nse3d": 4}.get(fam, 1)
    values = 2 * nf
    if fam == "srccde2d":
        values += 1 + case["steps"]
    size = 8 if case["storage"] == "fp64" else 4
    return {"bytes": nodes * values * size, "flops": nodes * case["steps"] * FLOPS[fam]}


# ------------------------------------------------------------------ 64-bit reference

def _lattice(fam):
    """(directions (x, y, z), weights) with c_s^2 = c^2 / 3 for D2Q9 and D3Q19."""
    if fam in DIM3:
        e, w = [(0, 0, 0)], [1 / 3]
        for x in (-1, 0, 1):
            for y in (-1, 0, 1):
                for z in (-1, 0, 1):
                    k = abs(x) + abs(y) + abs(z)
                    if k in (1, 2):
                        e.append((x, y, z))
                        w.append(1 / 18 if k == 1 else 1 / 36)
        return e, w
    e, w = [], []
    for x in (-1, 0, 1):
        for y in (-1, 0, 1):
            k = abs(x) + abs(y)
            e.append((x, y, 0))
            w.append((4 / 9, 1 / 9, 1 / 36)[k])
    return e, w


def _at(f, e, k):
    """f(x + k e) on the periodic grid."""
    dims, shifts = [], []
    for axis, v in enumerate(e):
        if v * k != 0:
            dims.append(f.dim() - 1 - axis)
            shifts.append(-v * k)
    return torch.roll(f, shifts, dims) if dims else f


def _add(acc, a, e, f):
    """acc += sum_k a_k f(x + k e), a = (a_{-1}, a_0, a_1)."""
    for k, v in zip((-1, 0, 1), a):
        if v != 0.0:
            acc.add_(_at(f, e, k), alpha=v)


def _linear_weights(case):
    """w_j of f_j = w_j phi for the linear PDEs, with the directions."""
    fam = case["family"]
    if fam == "cde3d":
        # axis lattice, linear EDF: c_s,a^2 = 2 K_a / dt - (A_21 - A_20 term), two levels, a = (1, 0, 0):
        # A_10 = -1, A_20 = 1/2, A_21 = 1, A_22 = 1/2
        e, w, rest = [], [], 1.0
        for axis in range(3):
            d0 = (K3[axis] + (1.0 - 0.5) * U3[axis] ** 2) / 0.5
            for s in (1, -1):
                v = [0, 0, 0]
                v[axis] = s
                e.append(tuple(v))
                w.append(d0 / 2 * (1 + s * U3[axis] / d0))
            rest -= d0
        return e + [(0, 0, 0)], w + [rest]
    e, w = _lattice(fam)
    if fam == "srccde2d":
        d, kappa = _src_scales(case)
        c, u, K, dt, a10, a22 = d["dx"] / d["dt"], (0.1, 0.1), [[kappa, 0], [0, kappa]], d["dt"], -1.0, 0.5
    else:
        dt = THETA_DT if fam == "theta2d" else 1.0
        c, u, K, a10, a22 = 1.0 / dt, U2, K2, -1.0, 0.5
    cs2 = c * c / 3
    C = [[-a10 * K[i][j] / (a22 * dt) + u[i] * u[j] - (cs2 if i == j else 0.0) for j in range(2)] for i in range(2)]
    out = []
    for ej, wj in zip(e, w):
        cj = (ej[0] * c, ej[1] * c)
        s = 1.0 + (cj[0] * u[0] + cj[1] * u[1]) / cs2
        for i in range(2):
            s += (cj[i] ** 2 - cs2) / (cs2 * (c * c - cs2)) * C[i][i]
        s += 2 * cj[0] * cj[1] / (2 * cs2 * cs2) * C[0][1]
        out.append(wj * s)
    return e, out


def _exact_linear(case, cur, prev, src):
    e, w = _linear_weights(case)
    three = case["family"] == "srccde2d"
    phi, old = cur[0], prev[0] if prev is not None else None
    last = None
    for m in range(case["steps"]):
        acc = torch.zeros_like(phi)
        for ej, wj in zip(e, w):
            if three:
                _add(acc, [v * wj for v in THREE_A], ej, phi)
                _add(acc, [v * wj for v in THREE_AHAT], ej, old)
            else:
                _add(acc, (wj, 0.0, 0.0), ej, phi)
        if src is not None:
            d, _ = _src_scales(case)
            c = d["dx"] / d["dt"]
            s = src[m][0].double()
            last = s if last is None else last
            es, ws = _lattice("srccde2d")
            for ej, wj in zip(es, ws):
                g = d["dt"] * wj * (1 + 3 * 0.1 * (ej[0] + ej[1]) / c)
                _add(acc, (1.5 * g, 0.0, 0.0), ej, s)
                _add(acc, (-0.5 * g, 0.0, 0.0), ej, last)
            last = s
        phi, old = acc, phi
    return [phi]


def _exact_theta(case, cur):
    e, w = _linear_weights(case)
    ny, nx = cur[0].shape
    kx = 2 * math.pi * torch.fft.rfftfreq(nx, dtype=torch.float64, device="cuda")[None, :]
    ky = 2 * math.pi * torch.fft.fftfreq(ny, dtype=torch.float64, device="cuda")[:, None]
    lam = torch.zeros(ny, nx // 2 + 1, dtype=torch.complex128, device="cuda")
    for ej, wj in zip(e, w):
        lam += wj * torch.exp(-1j * (ej[0] * kx + ej[1] * ky))
    lam -= 1.0
    lam = ((1 + 0.5 * lam) / (1 - 0.5 * lam)) ** case["steps"]
    return [torch.fft.irfft2(torch.fft.rfft2(cur[0]) * lam, s=(ny, nx))]


def _exact_ncde(case, cur):
    dx, dt = _ncde_scales(case)
    dim = 3 if case["family"] == "ncde3d" else 2
    c, (e, w) = dx / dt, _lattice(case["family"])
    cs2 = c * c / 3
    phi = old = cur[0]

    def parts(p):
        # B_a = p^2 / 2 and the isotropic second moment 2 G(p) / dt, G = 0.01 (p + p^3 / 3)
        m2 = (2 * 0.01 / dt) * (p + p ** 3 / 3)
        return 0.5 * p * p, m2 - cs2 * p

    for _ in range(case["steps"]):
        acc = torch.zeros_like(phi)
        for p, a in ((phi, THREE_A), (old, THREE_AHAT)):
            b, t = parts(p)
            for ej, wj in zip(e, w):
                q = sum(((ej[i] * c) ** 2 - cs2) / (cs2 * (c * c - cs2)) for i in range(dim))
                _add(acc, a, ej, wj * (p + (sum(ej) * c / cs2) * b + q * t))
        phi, old = acc, phi
    return [phi]


def _exact_nse(case, cur):
    e, w = _lattice(case["family"])
    dim = len(cur) - 1
    a0 = case["a0"]
    a, ab = (1.0, 0.0, 0.0), (1.0 - a0 / 2, a0, -a0 / 2)
    rho, u = cur[0], cur[1:]
    for _ in range(case["steps"]):
        new = [torch.zeros_like(rho) for _ in range(1 + dim)]
        # sum_a Q_aa u_a^2 of the rest direction, and per axis what a nonzero component adds
        half = -1.5 * sum(v * v for v in u)
        for ej, wj in zip(e, w):
            f = rho + half
            eu = None
            for i in range(dim):
                if ej[i]:
                    eu = ej[i] * u[i] if eu is None else eu + ej[i] * u[i]
            if eu is not None:
                # w (rho + 3 e.u + Q : uu) with Q_aa = (e_a^2 - 1/3) / (2/9), Q_ab = 9/2 e_a e_b
                f = f + 3 * eu + 4.5 * eu * eu
            f = wj * f
            _add(new[0], a, ej, f)
            for i in range(dim):
                if ej[i]:
                    _add(new[1 + i], [ej[i] * v for v in ab], ej, f)
        rho, u = new[0], new[1:]
    return [rho] + u


def exact(case, seed):
    cur, prev, src = _inputs(case, seed)
    cur = [f.double() for f in cur]
    prev = None if prev is None else [f.double() for f in prev]
    fam = case["family"]
    if fam == "theta2d":
        return _exact_theta(case, cur)
    if fam in ("nse2d", "nse3d"):
        return _exact_nse(case, cur)
    if fam in ("ncde2d", "ncde3d"):
        return _exact_ncde(case, cur)
    return _exact_linear(case, cur, prev, src)
