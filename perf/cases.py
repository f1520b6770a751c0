"""What the framework's users have it do, as cases that can be timed and checked.

A case is one call (or the few calls that belong together) of the public Python API: the stage
operator (`Solver.rhs`), CFL steps (`Solver.step`), a run to a time (`Solver.run`), independent
problems host to host (`Solver.pipeline`), the batched path (`Batch.step`) and the differentiable
rollout (`adjoint.rollout`, forward and backward).  Everything is FP64, the only type of the path.
Sizes are those of the repository's own workloads and tests, or generic odd ones of the same range.

`exact` is the scheme written plainly with torch tensors in 64 bits (whole arrays at a time, no
code of this package), differentiated by torch's autograd for the rollout.
"""
import math

import numpy as np
import torch

_DEV = "cuda"
_F64 = torch.float64
# operations per cell and SSP-RK3 step of the scheme as its formulas are written ((dim, system))
_FLOPS = {(1, "advection"): 1056, (1, "burgers"): 1065, (1, "euler"): 4641,
          (2, "advection"): 2169, (2, "burgers"): 2187, (2, "euler"): 13344}
_R2 = 4  # HWENO_FLAG_R2


def listed():
    return [
        # the scalar accuracy problem to its end time: 267 steps of 160 cells, launches and latency
        {"name": "run_advection1d_160", "entry": "run", "system": "advection", "dim": 1, "nx": 160, "ny": 1,
         "data": "sine", "bc": "periodic", "flags": 0, "t_end": 2.0},
        # a shock tube on the coarser of its two meshes: ten CFL steps from the host loop
        {"name": "step_euler1d_2048", "entry": "step", "system": "euler", "dim": 1, "nx": 2048, "ny": 1,
         "data": "riemann", "bc": "transmissive", "flags": 0, "steps": 10},
        # the same on the finer mesh, at an odd size
        {"name": "step_euler1d_16383", "entry": "step", "system": "euler", "dim": 1, "nx": 16383, "ny": 1,
         "data": "riemann", "bc": "transmissive", "flags": 0, "steps": 10},
        # one evaluation of the operator of a 2D scalar law on a ragged grid (a caller's own time stepper)
        {"name": "rhs_burgers2d_1021x517", "entry": "rhs", "system": "burgers", "dim": 2, "nx": 1021, "ny": 517,
         "data": "sine", "bc": "periodic", "flags": 0},
        # one evaluation of the 2D Euler operator across captured fronts, ragged, open boundaries
        {"name": "rhs_euler2d_fronts_517x389", "entry": "rhs", "system": "euler", "dim": 2, "nx": 517, "ny": 389,
         "data": "fronts", "bc": "transmissive", "flags": 0},
        # the two 2D Euler workloads: discontinuous at 1024^2, smooth at 4096^2 (the largest)
        {"name": "step_euler2d_quadrants_1024", "entry": "step", "system": "euler", "dim": 2, "nx": 1024, "ny": 1024,
         "data": "quadrants", "bc": "periodic", "flags": 0, "steps": 2},
        {"name": "step_euler2d_wave_4096", "entry": "step", "system": "euler", "dim": 2, "nx": 4096, "ny": 4096,
         "data": "wave", "bc": "periodic", "flags": 0, "steps": 1},
        # Rayleigh-Taylor (walls, fixed ends, gravity) on the middle of its three meshes
        {"name": "step_rt2d_120x480", "entry": "step", "system": "euler", "dim": 2, "nx": 120, "ny": 480,
         "data": "rt", "bc": "rt", "flags": 0, "steps": 5},
        # the per-cell characteristic bases (the faster variant users choose), ragged
        {"name": "step_euler2d_r2_1023x769", "entry": "step", "system": "euler", "dim": 2, "nx": 1023, "ny": 769,
         "data": "modes", "bc": "periodic", "flags": _R2, "steps": 2},
        # many uneven problems at once: the batched path
        {"name": "batch_40lines_4grids", "entry": "batch", "system": "euler", "dim": 2, "nx": 256, "ny": 256,
         "lines": 40, "grids": 4, "pick": 7, "steps": 2},
        # gradient of a rollout: two steps forward and backward through the autograd function
        {"name": "rollout_euler2d_512", "entry": "rollout", "system": "euler", "dim": 2, "nx": 512, "ny": 512,
         "data": "modes", "bc": "periodic", "flags": 0, "steps": 2},
        # independent problems from host memory to host memory
        {"name": "pipeline_euler2d_768", "entry": "pipeline", "system": "euler", "dim": 2, "nx": 768, "ny": 768,
         "data": "wave", "bc": "periodic", "flags": 0, "steps": 1, "count": 4},
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    entry = rng.choice(["run", "step1", "step1", "rhs", "rhs", "step2", "step2", "rt", "batch", "rollout", "pipeline"])
    if entry == "run":
        n = size(40, 640)
        return {"entry": "run", "system": rng.choice(["advection", "burgers"]), "dim": 1, "nx": n, "ny": 1,
                "data": "sine", "bc": "periodic", "flags": 0, "t_end": rng.uniform(0.1, 0.25)}
    if entry == "step1":
        return {"entry": "step", "system": "euler", "dim": 1, "nx": size(128, 16384), "ny": 1,
                "data": rng.choice(["riemann", "wave"]), "bc": "transmissive", "flags": 0, "steps": rng.randint(1, 10)}
    if entry == "rt":
        nx = size(40, 240)
        return {"entry": "step", "system": "euler", "dim": 2, "nx": nx, "ny": 4 * nx + rng.randint(-3, 3),
                "data": "rt", "bc": "rt", "flags": 0, "steps": rng.randint(1, 5)}
    if entry == "batch":
        side = rng.choice([128, 256, 320, 384])
        return {"entry": "batch", "system": "euler", "dim": 2, "nx": side, "ny": side, "lines": rng.randint(8, 64),
                "grids": rng.randint(0, 6), "pick": rng.randint(0, 10 ** 6), "steps": rng.randint(1, 3)}
    if entry == "rollout":
        return {"entry": "rollout", "system": "euler", "dim": 2, "nx": size(40, 512), "ny": size(40, 512),
                "data": rng.choice(["modes", "wave"]), "bc": "periodic", "flags": 0, "steps": rng.randint(1, 2)}
    if entry == "pipeline":
        return {"entry": "pipeline", "system": "euler", "dim": 2, "nx": size(128, 1024), "ny": size(128, 1024),
                "data": "wave", "bc": "periodic", "flags": 0, "steps": 1, "count": rng.randint(2, 5)}
    system = rng.choice(["advection", "burgers", "euler", "euler", "euler"])
    if system != "euler":
        data = rng.choice(["sine", "blocks"])
    else:
        data = rng.choice(["wave", "modes", "quadrants", "fronts"])
    bc = rng.choice(["periodic", "transmissive"] + (["reflective"] if system == "euler" else []))
    case = {"entry": entry[:4] if entry == "step2" else "rhs", "system": system, "dim": 2, "nx": size(48, 1600),
            "ny": size(48, 1600), "data": data, "bc": bc,
            "flags": _R2 if system == "euler" and rng.random() < 0.3 else 0}
    if entry == "step2":
        case["steps"] = rng.randint(1, 3)
    return case


# ---------------------------------------------------------------------------------------------
# inputs

def _conserved(prims, grads, gamma):
    """Planes (U, U_x[, U_y]) from primitive fields [rho, u[, v], p] and their derivatives."""
    rho, vel, p = prims[0], prims[1:-1], prims[-1]
    ke = sum(a * a for a in vel)
    out = [torch.stack([rho] + [rho * a for a in vel] + [p / (gamma - 1) + 0.5 * rho * ke])]
    for g in grads:
        dr, dv, dp = g[0], g[1:-1], g[-1]
        out.append(torch.stack([dr] + [dr * a + rho * da for a, da in zip(vel, dv)] +
                               [dp / (gamma - 1) + 0.5 * dr * ke + rho * sum(a * da for a, da in zip(vel, dv))]))
    return torch.stack(out)


def _box(case):
    """((x low, x high), (y low, y high)) of the problem's domain."""
    if case["data"] == "rt":
        return (0.0, 0.25), (0.0, 1.0)
    if case["data"] == "riemann":
        return (-5.0, 5.0), (0.0, 1.0)
    if case["system"] == "burgers":
        return ((-math.pi, math.pi),) * 2 if case["dim"] == 1 else ((-2 * math.pi, 2 * math.pi),) * 2
    return (0.0, 2.0), (0.0, 2.0)


def _spacing(case):
    (a, b), (c, d) = _box(case)
    dx = (b - a) / case["nx"]
    return dx, ((d - c) / case["ny"] if case["dim"] == 2 else dx)


def _gamma(case):
    return 5.0 / 3.0 if case.get("data") == "rt" else 1.4


def _state(case, seed):
    """The initial state (nfield, ncomp, ny, nx) on the GPU."""
    r = np.random.default_rng([int(seed), case["nx"], case["ny"]])
    nx, ny, dim, data, gamma = case["nx"], case["ny"], case["dim"], case["data"], _gamma(case)
    (a, b), (c, d) = _box(case)
    dx, dy = _spacing(case)
    x = (a + (torch.arange(nx, dtype=_F64, device=_DEV) + 0.5) * dx).reshape(1, nx)
    y = ((c + (torch.arange(ny, dtype=_F64, device=_DEV) + 0.5) * dy) if dim == 2
         else torch.zeros(1, dtype=_F64, device=_DEV)).reshape(ny, 1)
    zero = torch.zeros((ny, nx), dtype=_F64, device=_DEV)
    if case["system"] != "euler":
        if data == "blocks":  # piecewise constant, zero derivatives
            v = torch.tensor(r.uniform(-1.0, 2.0, 16), device=_DEV)
            ix = ((x - a) / (b - a) * 4).long().clamp(0, 3)
            iy = ((y - c) / (d - c) * 4).long().clamp(0, 3)
            return torch.stack([v[iy * 4 + ix]] + [zero] * dim)[:, None]
        k = math.pi if case["system"] == "advection" else (1.0 if dim == 1 else 0.5)
        s = k * (x + (y if dim == 2 else 0.0)) + r.uniform(0, 2 * math.pi) + zero
        amp = r.uniform(0.8, 1.0)
        der = amp * k * torch.cos(s)
        return torch.stack([0.5 + amp * torch.sin(s)] + [der] * dim)[:, None]
    ones = zero + 1.0
    if data == "riemann":
        (rl, rr), (ul, ur), (pl, pr) = r.uniform(0.1, 5, 2), r.uniform(-1, 1, 2), r.uniform(0.1, 10, 2)
        right = (x > r.uniform(-2, 2)) & (zero == 0)
        k = float(r.integers(1, 11))
        rho = torch.where(right, rr * (1 + 0.2 * torch.sin(k * x)), rl * ones)
        rx = torch.where(right, rr * 0.2 * k * torch.cos(k * x), zero)
        u, p = torch.where(right, ur * ones, ul * ones), torch.where(right, pr * ones, pl * ones)
        return _conserved([rho, u, p], [[rx, zero, zero]], gamma)
    if data == "quadrants":
        v = [torch.tensor(r.uniform(lo, hi, 4), device=_DEV) for lo, hi in ((0.1, 2), (-1, 1), (-1, 1), (0.1, 2))]
        q = (x >= 1.0).long() + 2 * (y >= 1.0).long()
        return _conserved([w[q] for w in v], [[zero] * 4] * 2, gamma)
    if data == "rt":
        rho = torch.where(y < 0.5, 2.0 * ones, ones)
        p = torch.where(y < 0.5, 2 * y + 1 + zero, y + 1.5 + zero)
        py = torch.where(y < 0.5, 2.0 * ones, ones)
        cs = torch.sqrt(gamma * p / rho)
        cy = 0.5 * gamma * py / (rho * cs)
        e = 0.025 * r.uniform(0.5, 1.0)
        cx, sx = torch.cos(8 * math.pi * x), torch.sin(8 * math.pi * x)
        return _conserved([rho, zero, -e * cs * cx, p], [[zero, zero, e * cs * 8 * math.pi * sx, zero],
                                                         [zero, zero, -e * cy * cx, py]], gamma)
    # the smooth wave, with seeded phase, amplitude and velocity, and modes or fronts upon it
    vel = [r.uniform(0.2, 0.8) * ones for _ in range(dim)]
    amp, ph = r.uniform(0.15, 0.25), r.uniform(0, 2 * math.pi)
    s = math.pi * (x + (y if dim == 2 else 0.0)) + ph + zero
    f = {"rho": [1 + amp * torch.sin(s)] + [amp * math.pi * torch.cos(s)] * dim, "p": [ones] + [zero] * dim}
    if data == "modes":  # eight modes of amplitude 0.05 / 8 each
        for name in ("rho", "p"):
            for _ in range(8):
                kx, ky = r.integers(1, 5), r.integers(-4, 5)
                arg = math.pi * (float(kx) * x + float(ky) * y) + r.uniform(0, 2 * math.pi)
                g = [0.00625 * torch.sin(arg), 0.00625 * math.pi * float(kx) * torch.cos(arg),
                     0.00625 * math.pi * float(ky) * torch.cos(arg)]
                f[name] = [o + n for o, n in zip(f[name], g)]
    if data == "fronts":  # five circular fronts about a cell wide, as a scheme captures them
        for _ in range(5):
            x0, y0, rad = r.uniform(0.2, 1.8), r.uniform(0.2, 1.8), r.uniform(0.2, 0.7)
            w = max(dx, dy)
            rr = torch.sqrt((x - x0) ** 2 + (y - y0) ** 2 + 1e-12)
            th = torch.tanh((rad - rr) / w)
            dth = -(1 - th * th) / (w * rr)
            for name, jump in (("rho", r.uniform(0.05, 0.3)), ("p", r.uniform(0.05, 0.5))):
                g = [jump * 0.5 * (1 + th), 0.5 * jump * dth * (x - x0), 0.5 * jump * dth * (y - y0)]
                f[name] = [o + n for o, n in zip(f[name], g)]
    return _conserved([f["rho"][0]] + vel + [f["p"][0]],
                      [[f["rho"][1 + k]] + [zero] * dim + [f["p"][1 + k]] for k in range(dim)], gamma)


_FIXED = {2: [2.0, 0.0, 0.0, 1.0 / (2.0 / 3.0)], 3: [1.0, 0.0, 0.0, 2.5 / (2.0 / 3.0)]}


def _solver(case):
    from paper_2411_11229_gb300 import Solver
    dx, dy = _spacing(case)
    more = dict(bc=case["bc"])
    if case["bc"] == "rt":
        more = dict(sides=("reflective", "reflective", "fixed", "fixed"), fixed=_FIXED, grav=1.0)
    return Solver(case["dim"], case["system"], case["nx"], case["ny"], dx=dx, dy=dy, gamma=_gamma(case),
                  flags=case["flags"], **more)


def _members(case):
    """The problems of a batch: lines of 128 to 8192 cells (log-uniform) and square grids."""
    r = np.random.default_rng(case["pick"])
    out = [{"dim": 1, "nx": int(round(math.exp(r.uniform(math.log(128), math.log(8192))))), "ny": 1,
            "system": "euler", "data": "riemann", "bc": "transmissive", "flags": 0} for _ in range(case["lines"])]
    return out + [{"dim": 2, "nx": case["nx"], "ny": case["ny"], "system": "euler", "bc": "periodic", "flags": 0,
                   "data": ("wave", "quadrants")[k % 2]} for k in range(case["grids"])]


def prepare(case, seed):
    st = {"case": case}
    if case["entry"] == "batch":
        from paper_2411_11229_gb300 import Batch
        ms = _members(case)
        descs = [dict(dim=m["dim"], nx=m["nx"], ny=m["ny"], dx=_spacing(m)[0], dy=_spacing(m)[1], bc=m["bc"])
                 for m in ms]
        st["batch"] = Batch(descs)
        st["S"] = torch.cat([_state(m, seed + 1000 * i).reshape(-1) for i, m in enumerate(ms)])
        return st
    st["solver"] = _solver(case)
    if case["entry"] == "pipeline":
        st["in"] = [_state(case, seed + 1000 * i).cpu().pin_memory() for i in range(case["count"])]
        st["out"] = [torch.empty_like(t).pin_memory() for t in st["in"]]
        return st
    st["S"] = _state(case, seed)
    if case["entry"] == "rollout":
        st["S"].requires_grad_(True)
        st["area"] = math.prod(_spacing(case))
    return st


def run(st):
    case = st["case"]
    entry = case["entry"]
    if entry == "batch":
        b = st["batch"]
        with torch.cuda.stream(b.stream):
            b.stream.wait_stream(torch.cuda.default_stream())
            b.state.copy_(st["S"])
        b.step(case["steps"])
        torch.cuda.current_stream().wait_stream(b.stream)
        return b.state
    s = st["solver"]
    if entry == "rhs":
        L, M = s.rhs(st["S"])
        return {"L": L, "M": M}
    if entry == "step":
        s.set_state(st["S"])
        s.step(0.0, case["steps"])
        return s.state
    if entry == "run":
        s.set_state(st["S"])
        n = s.run(case["t_end"])
        return {"state": s.state, "steps": n}
    if entry == "pipeline":
        s.pipeline(st["in"], st["out"], nsteps=case["steps"], depth=3)
        return st["out"]
    from paper_2411_11229_gb300.adjoint import rollout
    st["S"].grad = None
    ST = rollout(st["S"], s, case["steps"], keep_stages=True)
    (0.5 * (ST[0, 0] ** 2).sum() * st["area"]).backward()
    return {"state": ST.detach(), "grad": st["S"].grad}


def work(case):
    """Inputs read once and outputs written once; the operations of the scheme's formulas."""
    if case["entry"] == "batch":
        ms = _members(case)
        cells = sum(m["nx"] * m["ny"] * (6 if m["dim"] == 1 else 12) for m in ms)
        flops = sum(m["nx"] * m["ny"] * _FLOPS[(m["dim"], "euler")] for m in ms)
        return {"bytes": 16.0 * cells, "flops": float(flops * case["steps"])}
    dim, cells = case["dim"], case["nx"] * case["ny"]
    values = cells * (dim + 1) * ((dim + 2) if case["system"] == "euler" else 1)
    flops = _FLOPS[(dim, case["system"])] * cells
    entry = case["entry"]
    if entry == "rhs":
        return {"bytes": 24.0 * values, "flops": flops / 3.0}
    if entry == "run":  # CFL 0.6 and wavespeeds about 1 (advection) and 1.5 (Burgers)
        speed = 1.0 if case["system"] == "advection" else 1.45
        return {"bytes": 16.0 * values, "flops": flops * math.ceil(case["t_end"] * speed / (0.6 * _spacing(case)[0]))}
    if entry == "pipeline":
        return {"bytes": 16.0 * values * case["count"], "flops": float(flops * case["steps"] * case["count"])}
    if entry == "rollout":  # the reverse of a step holds the step's operations and their transposes
        return {"bytes": 24.0 * values, "flops": 3.0 * flops * case["steps"]}
    return {"bytes": 16.0 * values, "flops": float(flops * case["steps"])}


# ---------------------------------------------------------------------------------------------
# the scheme in plain torch, 64 bits: fields [component, line, along] in the sweep's own frame

def _weights(dm, dp, hm, hp, eps):
    """1 + tau / (beta_l + eps) of the stencil with differences dm, dp and end slopes hm, hp (times h)."""
    du, d2, sv, dv = dm + dp, dp - dm, hm + hp, hm - hp
    b0 = ((11 / 16) * du - (3 / 16) * sv) ** 2 + (13 / 3) * ((67 / 520) * dv + (197 / 260) * d2) ** 2 \
        + (781 / 20) * (0.25 * (sv - du)) ** 2 + (1421461 / 2275) * (0.25 * (dv + 2 * d2)) ** 2
    b1, b2 = dm * dm, dp * dp
    tau = (0.5 * ((b0 - b1).abs() + (b0 - b2).abs())) ** 2
    return [1 + tau / (b + eps) for b in (b0, b1, b2)]


def _interp(dm, dp, hm, hp, g0, eps):
    """The value at the stencil's right face less the centre value."""
    g1 = 0.5 * (1 - g0)
    W = _weights(dm, dp, hm, hp, eps)
    p0 = 0.125 * dm + 0.5625 * dp - 0.046875 * hm - 0.140625 * hp
    p1, p2 = 0.5 * dm, 0.5 * dp
    return (W[0] * (p0 - g1 * (p1 + p2)) + g1 * (W[1] * p1 + W[2] * p2)) / (g0 * W[0] + g1 * (W[1] + W[2]))


def _limit(dm, dp, hm, hp, eps, d0=0.9):
    """h times the modified derivative at the centre."""
    d1 = 0.5 * (1 - d0)
    W = _weights(dm, dp, hm, hp, eps)
    q0 = 0.75 * (dm + dp) - 0.25 * (hm + hp)
    return (W[0] * (q0 - d1 * (dm + dp)) + d1 * (W[1] * dm + W[2] * dp)) / (d0 * W[0] + d1 * (W[1] + W[2]))


def _prim(U, gamma):
    vel = [U[k] / U[0] for k in range(1, len(U) - 1)]
    ke = 0.5 * U[0] * sum(a * a for a in vel)
    return vel, (gamma - 1) * (U[-1] - ke)


def _basis(vel, H, c, gamma):
    """Left and right products with the eigenvectors of the sweep's Jacobian."""
    u, q2 = vel[0], 0.5 * sum(a * a for a in vel)
    b1 = (gamma - 1) / (c * c)

    def left(q):
        t = b1 * (q2 * q[0] - sum(a * m for a, m in zip(vel, q[1:-1])) + q[-1])
        s = (u * q[0] - q[1]) / c
        shear = [q[2] - vel[1] * q[0]] if len(vel) == 2 else []
        return torch.stack([0.5 * (t + s), q[0] - t] + shear + [0.5 * (t - s)])

    def right(w):
        sg, dl = w[0] + w[-1], w[-1] - w[0]
        q0 = sg + w[1]
        out = [q0, u * q0 + c * dl]
        last = H * sg + q2 * w[1] + u * c * dl
        if len(vel) == 2:
            out.append(vel[1] * q0 + w[2])
            last = last + vel[1] * w[2]
        return torch.stack(out + [last])

    return left, right


class _Law:
    def __init__(self, case):
        self.system, self.gamma = case["system"], _gamma(case)
        self.r2 = bool(case.get("flags", 0) & _R2) and self.system == "euler"
        self.g0 = 0.95 if case["dim"] == 1 else 0.99

    def flux(self, U):
        if self.system == "advection":
            return U
        if self.system == "burgers":
            return 0.5 * U * U
        vel, p = _prim(U, self.gamma)
        shear = [U[2] * vel[0]] if len(vel) == 2 else []
        return torch.stack([U[1], U[1] * vel[0] + p] + shear + [(U[-1] + p) * vel[0]])

    def jvp(self, U, D):
        if self.system == "advection":
            return D
        if self.system == "burgers":
            return U * D
        vel, p = _prim(U, self.gamma)
        dv = [(D[1 + k] - a * D[0]) / U[0] for k, a in enumerate(vel)]
        dk = sum(D[1 + k] * a + U[1 + k] * d for k, (a, d) in enumerate(zip(vel, dv)))
        dp = (self.gamma - 1) * (D[-1] - 0.5 * dk)
        shear = [D[2] * vel[0] + U[2] * dv[0]] if len(vel) == 2 else []
        return torch.stack([D[1], D[1] * vel[0] + U[1] * dv[0] + dp] + shear +
                           [(D[-1] + dp) * vel[0] + (U[-1] + p) * dv[0]])

    def speed(self, U):
        if self.system == "advection":
            return torch.ones_like(U[0])
        if self.system == "burgers":
            return U[0].abs()
        vel, p = _prim(U, self.gamma)
        return vel[0].abs() + torch.sqrt(self.gamma * p / U[0])

    def own_basis(self, U):
        vel, p = _prim(U, self.gamma)
        return _basis(vel, (U[-1] + p) / U[0], torch.sqrt(self.gamma * p / U[0]), self.gamma)

    def roe_basis(self, A, B):
        (va, pa), (vb, pb) = _prim(A, self.gamma), _prim(B, self.gamma)
        a, b = torch.sqrt(A[0]), torch.sqrt(B[0])
        mean = lambda s, t: (a * s + b * t) / (a + b)  # noqa: E731
        vel = [mean(s, t) for s, t in zip(va, vb)]
        H = mean((A[-1] + pa) / A[0], (B[-1] + pb) / B[0])
        return _basis(vel, H, torch.sqrt((self.gamma - 1) * (H - 0.5 * sum(s * s for s in vel))), self.gamma)

    def sweep(self, U, D, O, ends, h, alpha, eps=1e-10):
        """Flux differences of U, D, O over h along the last axis, and the modified derivative."""
        U, D, O = _ghosts(U, D, O, ends)
        n = U.shape[-1] - 4
        c = lambda F, q: F[..., q:q + n + 1]  # noqa: E731  cells fa-2+q of the faces
        d = [c(U, q + 1) - c(U, q) for q in range(3)]
        y = [h * c(D, q) for q in range(4)]
        if self.system != "euler":
            ident = (lambda w: w, lambda w: w)
            bm = bp = ident
        elif self.r2:
            bm, bp = self.own_basis(c(U, 1)), self.own_basis(c(U, 2))
        else:
            bm = bp = self.roe_basis(c(U, 1), c(U, 2))
        Um = c(U, 1) + bm[1](_interp(bm[0](d[0]), bm[0](d[1]), bm[0](y[0]), bm[0](y[2]), self.g0, eps))
        Up = c(U, 2) + bp[1](_interp(-bp[0](d[2]), -bp[0](d[1]), -bp[0](y[3]), -bp[0](y[1]), self.g0, eps))
        Dm = (1.3125 * d[1] - 0.1875 * d[0] + 0.0625 * y[0] - 0.1875 * y[2]) / h
        Dp = (1.3125 * d[1] - 0.1875 * d[2] - 0.1875 * y[1] + 0.0625 * y[3]) / h
        f, g = self.flux(U), self.jvp(U, D)
        f0, f1, f2, f3 = (c(f, q) for q in range(4))
        ga, gb = c(g, 0), c(g, 3)
        # the second and fourth derivatives of the degree-5 central Hermite interpolant, times h^2, h^4
        s = (f0 - f1) + (f3 - f2)
        Df = -(1 / 24) * ((9 / 8) * s + (5 / 12) * h * (ga - gb)) + (7 / 5760) * (-3 * s - 2 * h * (ga - gb))
        Dh = ((1 / 24) * ((101 / 36) * (f0 - f3) + (27 / 4) * (f2 - f1)) +
              (7 / 5760) * ((130 / 9) * (f0 - f3) + 30 * (f2 - f1))) / h + \
            ((1 / 24) * (5 / 6) + (7 / 5760) * (20 / 3)) * (ga + gb)
        fh = 0.5 * (self.flux(Um) + self.flux(Up) - alpha * (Up - Um)) + Df
        hh = 0.5 * (self.jvp(Um, Dm) + self.jvp(Up, Dp) - alpha * (Dp - Dm)) + Dh
        L = [-(fh[..., 1:] - fh[..., :-1]) / h, -(hh[..., 1:] - hh[..., :-1]) / h, None]
        if O is not None:
            o = self.jvp(U, O)
            oh = (7 / 12) * (c(o, 1) + c(o, 2)) - (1 / 12) * (c(o, 0) + c(o, 3))
            L[2] = -(oh[..., 1:] - oh[..., :-1]) / h
        i = lambda F, q: F[..., 1 + q:1 + q + n]  # noqa: E731  cells i-1+q
        dm, dp, hm, hp = i(U, 1) - i(U, 0), i(U, 2) - i(U, 1), h * i(D, 0), h * i(D, 2)
        b = self.own_basis(i(U, 1)) if self.system == "euler" else (lambda w: w, lambda w: w)
        return L, b[1](_limit(b[0](dm), b[0](dp), b[0](hm), b[0](hp), eps)) / h


def _ghosts(U, D, O, ends):
    """Two ghost cells at both ends of the last axis; ends: a type, or a fixed state, for each."""
    fields = [U, D] + ([O] if O is not None else [])
    lo, hi = [], []
    for f, F in enumerate(fields):
        sides = []
        for e, kind in enumerate(ends):
            if kind == "periodic":
                g = F[..., -2:] if e == 0 else F[..., :2]
            elif kind == "transmissive":
                g = (F[..., :1] if e == 0 else F[..., -1:]).expand(*F.shape[:-1], 2)
            elif kind == "reflective":
                g = (F[..., :2] if e == 0 else F[..., -2:]).flip(-1)
                s = torch.ones(F.shape[0], dtype=F.dtype, device=F.device)
                s[1] = -1.0
                g = g * (-s if f == 1 else s)[:, None, None]
            else:
                g = torch.tensor(kind, dtype=F.dtype, device=F.device)[:, None, None] * (1.0 if f == 0 else 0.0)
                g = g.expand(*F.shape[:-1], 2)
            sides.append(g)
        lo.append(sides[0])
        hi.append(sides[1])
    out = [torch.cat([a, F, b], -1) for a, F, b in zip(lo, fields, hi)]
    return out[0], out[1], (out[2] if O is not None else None)


def _turn(F):
    """A field [component, y, x] in the frame of the y sweep: [component, x, y], momenta exchanged."""
    F = F.transpose(-1, -2)
    return F[[0, 2, 1, 3]] if F.shape[0] == 4 else F


def _ends(case, direction):
    if case["bc"] != "rt":
        return (case["bc"],) * 2
    return ("reflective",) * 2 if direction == 0 else tuple([v[0], v[2], v[1], v[3]] for v in (_FIXED[2], _FIXED[3]))


def _alphas(law, S):
    ax = law.speed(S[0]).max().detach()
    return (ax, law.speed(_turn(S[0])).max().detach()) if len(S) == 3 else (ax, None)


def _rhs(case, law, S, alpha):
    dx, dy = _spacing(case)
    if case["dim"] == 1:
        L, v = law.sweep(S[0], S[1], None, _ends(case, 0), dx, alpha[0])
        return torch.stack(L[:2]), torch.stack([S[0], v])
    (a, b, c), v = law.sweep(S[0], S[1], S[2], _ends(case, 0), dx, alpha[0])
    (p, q, r), w = law.sweep(_turn(S[0]), _turn(S[2]), _turn(S[1]), _ends(case, 1), dy, alpha[1])
    L = [a + _turn(p), b + _turn(r), c + _turn(q)]
    if case["bc"] == "rt":  # gravity g = 1 along +y
        z = torch.zeros_like(S[0][0])
        L = [f + torch.stack([z, z, F[0], F[2]]) for f, F in zip(L, S)]
    return torch.stack(L), torch.stack([S[0], v, _turn(w)])


def _step(case, law, S, left=None):
    """One SSP-RK3 step at CFL 0.6 (at most `left`): the new state and dt."""
    dx, dy = _spacing(case)
    al = _alphas(law, S)
    dt = 0.6 * dx / al[0] if case["dim"] == 1 else 0.6 / (al[0] / dx + al[1] / dy)
    if left is not None:
        dt = torch.clamp(dt, max=left)
    L, M0 = _rhs(case, law, S, al)
    S1 = M0 + dt * L
    L, M = _rhs(case, law, S1, _alphas(law, S1))
    S2 = 0.75 * M0 + 0.25 * (M + dt * L)
    L, M = _rhs(case, law, S2, _alphas(law, S2))
    return M0 / 3 + (2 / 3) * (M + dt * L), float(dt)


def exact(case, seed):
    entry = case["entry"]
    if entry == "batch":
        out = []
        for i, m in enumerate(_members(case)):
            S, law = _state(m, seed + 1000 * i), _Law(m)
            for _ in range(case["steps"]):
                S, _ = _step(m, law, S)
            out.append(S.reshape(-1))
        return torch.cat(out)
    law = _Law(case)
    if entry == "pipeline":
        out = []
        for i in range(case["count"]):
            S = _state(case, seed + 1000 * i)
            for _ in range(case["steps"]):
                S, _ = _step(case, law, S)
            out.append(S.cpu())
        return out
    S = _state(case, seed)
    if entry == "rhs":
        L, M = _rhs(case, law, S, _alphas(law, S))
        return {"L": L, "M": M}
    if entry == "run":
        t, n = 0.0, 0
        while t < case["t_end"]:
            S, dt = _step(case, law, S, case["t_end"] - t)
            t, n = t + dt, n + 1
        return {"state": S, "steps": n}
    if entry == "step":
        for _ in range(case["steps"]):
            S, _ = _step(case, law, S)
        return S
    S.requires_grad_(True)
    T = S
    for _ in range(case["steps"]):
        T, _ = _step(case, law, T)
    (0.5 * (T[0, 0] ** 2).sum() * math.prod(_spacing(case))).backward()
    return {"state": T.detach(), "grad": S.grad}
