"""What this framework is used for, as measurable passes through its public entry points.

A pass of a D2Q9 or D3Q27 case is what a user's program does with a lattice it
keeps: set the start fields, advance some steps, read density and velocity.
The sizes are those of the configurations, the experiments and the benchmark of
this repository; ``draw`` spreads more cases over the same ranges.
"""
from __future__ import annotations

import math

import numpy as np
import torch
import torch.utils.checkpoint

from paper_1202_6351_gb300 import adjoint, lbm

STORES = {"f64": lbm.F64, "f32": lbm.F32, "bf16": lbm.BF16DEV, "f16": lbm.F16DEV}
BYTES = {"f64": 8, "f32": 4, "bf16": 2, "f16": 2}
MODELS = {"cascaded": lbm.CASCADED, "bgk": lbm.BGK, "rawmrt": lbm.RAWMRT}
P, BB, MW = lbm.PERIODIC, lbm.BOUNCEBACK, lbm.MOVING_WALL
EDGES = {"periodic": (P, P, P, P), "channel": (P, P, BB, BB), "cavity": (BB, BB, BB, MW)}
LID = 0.1  # speed of the moving north wall of a cavity
# floating-point operations of one lattice update (additions and products of the
# moments, the relaxation and the back-transform), one direction; a reverse step
# of the adjoint recomputes the forward one and walks it backwards
FLOPS_2D, FLOPS_3D, FLOPS_ADJOINT = 150, 800, 650


def _flow(nx, ny, steps, store="f32", model="cascaded", edges="periodic", force="none", rounding="nearest",
          variant=-1, check=0, populations=False):
    return {"kind": "flow", "nx": nx, "ny": ny, "steps": steps, "store": store, "model": model,
            "edges": edges, "force": force, "rounding": rounding, "variant": variant, "check": check,
            "populations": populations}


def _flow3(nx, ny, nz, steps, store, force):
    return {"kind": "flow3", "nx": nx, "ny": ny, "nz": nz, "steps": steps, "store": store, "force": force}


def _gradient(nx, ny, steps, every, store):
    return {"kind": "gradient", "nx": nx, "ny": ny, "steps": steps, "every": every, "store": store}


def _ensemble(count, side_min, side_max, steps, pick, two_step):
    return {"kind": "ensemble", "count": count, "side_min": side_min, "side_max": side_max,
            "steps": steps, "pick": pick, "two_step": two_step}


def listed():
    return [
        # Poiseuille channel of the validation runs: the smallest lattice, FP64, driven by
        # a uniform force, thousands of steps; the populations are kept as a checkpoint
        {"name": "channel_f64_4x32"} | _flow(4, 32, 1000, store="f64", edges="channel", force="uniform", populations=True),
        # cavity of the stability and grid-convergence experiments, which step a thousand
        # steps at a time with the divergence check on
        {"name": "cavity_check_f32_101"} | _flow(101, 101, 1000, edges="cavity", check=1000),
        # the cavity configuration with a sibling collision run side by side with the cascaded one
        {"name": "cavity_rawmrt_f32_257"} | _flow(257, 257, 500, model="rawmrt", edges="cavity"),
        # decaying periodic flow on a middle-sized lattice that stays in the L2 cache
        {"name": "periodic_f32_512"} | _flow(512, 512, 500),
        # the cavity configuration's finest grid in 16-bit storage
        {"name": "cavity_f16_1025"} | _flow(1025, 1025, 200, store="f16", edges="cavity"),
        # the benchmark's flow: FP32, two steps per launch, 100 steps between transfers
        {"name": "periodic_f32_4096"} | _flow(4096, 4096, 100, variant=3),
        # a long 16-bit run at stated accuracy: stochastic rounding, an odd number of steps
        {"name": "periodic_f16_sr_2048"} | _flow(2048, 2048, 101, store="f16", rounding="stochastic"),
        # a large cavity in 16-bit storage, the roofline point of the 16-bit kernels
        {"name": "cavity_f16_8192"} | _flow(8192, 8192, 64, store="f16", edges="cavity"),
        # three-dimensional periodic flow, host fields in and out
        {"name": "d3q27_f32_192"} | _flow3(192, 192, 192, 200, "f32", False),
        # the same in 16-bit storage on a ragged box, with a body force
        {"name": "d3q27_f16_forced_127x96x130"} | _flow3(127, 96, 130, 300, "f16", True),
        # gradients of a final-state loss with respect to start field, force field and shear rate
        {"name": "gradient_f32_512"} | _gradient(512, 512, 400, 100, "f32"),
        # an ensemble of independent lattices of mixed sizes, edges and storage in one batch
        {"name": "ensemble_24"} | _ensemble(24, 64, 2048, 100, 1, True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["flow"] * 6 + ["flow3", "flow3", "gradient", "ensemble"])
    if kind == "flow3":
        nx, ny, nz = (_log_int(rng, 24, 192) for _ in range(3))
        return _flow3(nx, ny, nz, rng.randint(100, 200), rng.choice(["f32", "f32", "f16", "bf16"]),
                      rng.random() < 0.5)
    if kind == "gradient":
        every = rng.choice([25, 50, 100])
        return _gradient(_log_int(rng, 64, 512), _log_int(rng, 64, 512), rng.randint(50, 400), every, "f32")
    if kind == "ensemble":
        lo = _log_int(rng, 32, 128)
        return _ensemble(rng.randint(2, 24), lo, lo * rng.choice([4, 8, 16]), rng.randint(50, 100),
                         rng.randint(2, 1 << 20), rng.random() < 0.7)
    store = rng.choice(["f32", "f32", "f32", "f16", "f16", "bf16", "f64"])
    hi = 256 if store == "f64" else 4096
    nx, ny = _log_int(rng, 16, hi), _log_int(rng, 16, hi)
    most = 5e6 if store == "f64" else 4e9
    steps = max(11, min(_log_int(rng, 50, 1000), int(most / (nx * ny))))
    rounding = "stochastic" if store != "f64" and rng.random() < 0.25 else "nearest"
    return _flow(nx, ny, steps, store, rng.choice(["cascaded", "cascaded", "cascaded", "bgk", "rawmrt"]),
                 rng.choice(["periodic", "cavity", "channel"]), rng.choice(["none", "none", "uniform", "field"]),
                 rounding, rng.choice([-1, -1, 3]) if store != "f64" else -1, rng.choice([0, 0, 0, steps]),
                 nx * ny <= 1 << 16)


# ---------------------------------------------------------------- inputs

def _modes(seed, shape, amp, count=12, kmax=6):
    """Smooth divergence-free velocity [d, *shape] of `count` random Fourier modes (max |u| = amp) and a
    density near 1, float64 on the GPU; shape = (ny, nx) or (nz, ny, nx)."""
    rng = np.random.default_rng(seed)
    axes = [torch.arange(n, dtype=torch.float64, device="cuda") * (2.0 * math.pi / n) for n in shape]
    grid = [a.reshape([-1 if i == j else 1 for j in range(len(shape))]) for i, a in enumerate(axes)][::-1]  # x, y(, z)
    n_of = list(shape)[::-1]
    d = len(shape)
    u = torch.zeros((d,) + tuple(shape), dtype=torch.float64, device="cuda")
    rho = torch.ones(tuple(shape), dtype=torch.float64, device="cuda")
    for _ in range(count):
        k = [0] * d
        while not any(k):
            k = [int(v) for v in rng.integers(-kmax, kmax + 1, size=d)]
        kv = np.array([k[i] / n_of[i] for i in range(d)])
        a = rng.standard_normal(d)
        a -= kv * (a @ kv) / (kv @ kv)  # transverse: divergence-free
        phase = float(rng.uniform(0.0, 2.0 * math.pi))
        arg = sum(float(k[i]) * grid[i] for i in range(d)) + phase
        s = torch.sin(arg)
        for i in range(d):
            u[i] += float(a[i]) * s
        rho += 1e-4 * float(rng.standard_normal()) * torch.cos(arg)
    peak = float(u.square().sum(0).max().sqrt())
    if peak > 0.0:
        u *= amp / peak
    return rho, u


def _rates(nu):
    w = 1.0 / (3.0 * nu + 0.5)
    return (1.0, w, w, 1.0, 1.0, 1.0)


def _domains(case):
    """Sides, edges, storage and rates of an ensemble's lattices (half cavities, half periodic, FP32 and FP16)."""
    rng = np.random.default_rng(20261202 + case["pick"])
    out = []
    for i in range(case["count"]):
        n = int(round(math.exp(rng.uniform(math.log(case["side_min"]), math.log(case["side_max"])))))
        nu = max(LID * n / float(rng.uniform(100.0, 5000.0)), 0.002)
        out.append((n, "cavity" if i % 2 == 0 else "periodic", "f32" if (i // 2) % 2 == 0 else "f16", _rates(nu)))
    return out


def _flow_inputs(case, seed):
    ny, nx = case["ny"], case["nx"]
    rho, u = _modes(seed, (ny, nx), 0.04)
    force = (2e-6, 1e-6) if case["force"] == "uniform" else (0.0, 0.0)
    field = 1e-6 * _modes(seed + 1, (ny, nx), 1.0)[1].contiguous() if case["force"] == "field" else None
    # Re 1000 on the longer side, kept away from the stability limit of the siblings
    rates = _rates(max(LID * max(nx, ny) / 1000.0, 0.02))
    return rho, u, force, field, rates


def _flow3_inputs(case, seed):
    rho, u = _modes(seed, (case["nz"], case["ny"], case["nx"]), 0.04)
    w = 1.0 / (3.0 * 0.02 + 0.5)
    return rho, u, (1e-6, -2e-6, 1e-6) if case["force"] else (0.0, 0.0, 0.0), (1.0, w, 1.0, 1.0, 1.0, 1.0)


def _gradient_inputs(case, seed):
    shape = (case["ny"], case["nx"])
    return (_modes(seed, shape, 0.02)[1].contiguous(), 1e-6 * _modes(seed + 1, shape, 1.0)[1].contiguous(),
            _modes(seed + 2, shape, 0.02)[1].contiguous(), 1.6)


def prepare(case, seed):
    stream = torch.cuda.current_stream().cuda_stream
    if case["kind"] == "flow":
        rho, u, force, field, rates = _flow_inputs(case, seed)
        L = lbm.Lattice(case["nx"], case["ny"], rates, force=force, edges=EDGES[case["edges"]],
                        wall_u=(0.0, 0.0, 0.0, LID if case["edges"] == "cavity" else 0.0), model=MODELS[case["model"]],
                        store=STORES[case["store"]], stream=stream)
        if field is not None:
            L.set_force_field(field)
        if case["rounding"] == "stochastic":
            L.set_rounding(lbm.ROUND_STOCHASTIC, seed)
        if case["variant"] >= 0:
            L.set_variant(case["variant"])
        if case["check"]:
            L.set_check(case["check"], 1e-3)
        return {"case": case, "lattice": L, "rho": rho, "u": u}
    if case["kind"] == "flow3":
        rho, u, force, rates = _flow3_inputs(case, seed)
        L = lbm.Lattice3(case["nx"], case["ny"], case["nz"], rates, force=force, store=STORES[case["store"]],
                         stream=stream)
        return {"case": case, "lattice": L, "rho": rho.cpu().numpy(), "u": u.cpu().numpy()}
    if case["kind"] == "gradient":
        u0, force, target, omega = _gradient_inputs(case, seed)
        return {"case": case, "u0": u0.requires_grad_(), "force": force.requires_grad_(), "target": target,
                "omega": torch.tensor(omega, dtype=torch.float64, device="cuda", requires_grad=True)}
    lattices, fields = [], []
    for i, (n, edges, store, rates) in enumerate(_domains(case)):
        lattices.append(lbm.Lattice(n, n, rates, edges=EDGES[edges],
                                    wall_u=(0.0, 0.0, 0.0, LID if edges == "cavity" else 0.0),
                                    store=STORES[store], stream=stream))
        fields.append(_modes(seed + 1000 * i, (n, n), 0.04))
    B = lbm.Batch(lattices)
    if case["two_step"]:
        B.set_two_step(True)
    return {"case": case, "lattices": lattices, "fields": fields, "batch": B}


def run(state):
    case = state["case"]
    if case["kind"] == "flow":
        L = state["lattice"]
        L.init_device(state["rho"], state["u"])
        L.step(case["steps"])
        out = list(L.macros_device())
        if case["populations"]:
            out.append(L.get_f_device())
        return out
    if case["kind"] == "flow3":
        L = state["lattice"]
        L.init(state["rho"], state["u"])
        L.step(case["steps"])
        return list(L.macros())
    if case["kind"] == "gradient":
        u0, force, omega = state["u0"], state["force"], state["omega"]
        loss = adjoint.final_velocity_loss(u0, force, omega, state["target"], case["steps"], case["every"],
                                           store=STORES[case["store"]])
        return [loss.detach()] + list(torch.autograd.grad(loss, (u0, force, omega)))
    for L, (rho, u) in zip(state["lattices"], state["fields"]):
        L.init_device(rho, u)
    state["batch"].step(case["steps"])
    out = []
    for L in state["lattices"]:
        out += list(L.macros_device())
    return out


def work(case):
    """Each start field read once and each result written once (float64), and the updates' operations."""
    if case["kind"] == "flow":
        n = case["nx"] * case["ny"]
        fields = 6 + (9 if case["populations"] else 0) + (2 if case["force"] == "field" else 0)
        return {"bytes": 8 * fields * n, "flops": FLOPS_2D * n * case["steps"]}
    if case["kind"] == "flow3":
        n = case["nx"] * case["ny"] * case["nz"]
        return {"bytes": 8 * 8 * n, "flops": FLOPS_3D * n * case["steps"]}
    if case["kind"] == "gradient":
        n = case["nx"] * case["ny"]
        return {"bytes": 8 * 10 * n, "flops": (FLOPS_2D + FLOPS_ADJOINT) * n * case["steps"]}
    n = sum(d[0] * d[0] for d in _domains(case))
    return {"bytes": 8 * 6 * n, "flops": FLOPS_2D * n * case["steps"]}


# ---------------------------------------------------------------- the same in 64 bits, in plain torch

_E = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
_OPP = [0, 3, 4, 1, 2, 7, 8, 5, 6]
_W = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
# orthogonal basis of the raw-moment collision, rows = moments
_K = [[1] * 9, [e[0] for e in _E], [e[1] for e in _E], [3 * (e[0] ** 2 + e[1] ** 2) - 4 for e in _E],
      [e[0] ** 2 - e[1] ** 2 for e in _E], [e[0] * e[1] for e in _E],
      [-3 * e[0] ** 2 * e[1] + 2 * e[1] for e in _E], [-3 * e[0] * e[1] ** 2 + 2 * e[0] for e in _E],
      [9 * e[0] ** 2 * e[1] ** 2 - 6 * (e[0] ** 2 + e[1] ** 2) + 4 for e in _E]]


def _forward(f, u, dim):
    """Values at e = -1, 0, 1 along axis `dim` to central moments of order 0, 1, 2 about u."""
    a, b, c = f.unbind(dim)
    k0, s, p = a + b + c, c - a, c + a
    return torch.stack([k0, s - u * k0, p - 2 * u * s + u * u * k0], dim)


def _inverse(k, u, dim):
    k0, k1, k2 = k.unbind(dim)
    r1 = k1 + u * k0
    r2 = k2 + 2 * u * k1 + u * u * k0
    return torch.stack([0.5 * (r2 - r1), k0 - r2, 0.5 * (r2 + r1)], dim)


def _grid(f):  # paper order -> [e_x + 1][e_y + 1]
    return torch.stack([torch.stack([f[_E.index((x, y))] for y in (-1, 0, 1)]) for x in (-1, 0, 1)])


def _paper(g):
    return torch.stack([g[x + 1, y + 1] for x, y in _E])


def _from_central(k, u):
    return _paper(_inverse(_inverse(k, u[1], 1), u[0], 0))


def _equilibrium(model, rho, u):
    if model == "cascaded":
        z = torch.zeros_like(rho)
        m = [1.0, 0.0, 1 / 3]
        return _from_central(torch.stack([torch.stack([rho * (m[i] * m[j]) + z for j in range(3)]) for i in range(3)]), u)
    usq = u[0] ** 2 + u[1] ** 2
    out = []
    for (x, y), w in zip(_E, _W):
        eu = x * u[0] + y * u[1]
        out.append(w * rho * (1 + 3 * eu + 4.5 * eu * eu - 1.5 * usq))
    return torch.stack(out)


def _source(u, F):
    z = torch.zeros_like(u[0])
    k = [[z, F[1] + z, z], [F[0] + z, z, z], [z, z, z]]
    return _from_central(torch.stack([torch.stack(r) for r in k]), u)


def _macros(f, F):
    rho = f.sum(0)
    j = torch.stack([sum(e[i] * f[q] for q, e in enumerate(_E) if e[i]) for i in range(2)])
    return rho, torch.stack([(j[0] + 0.5 * F[0]) / rho, (j[1] + 0.5 * F[1]) / rho])


def _collide(model, f, F, om, forced):
    rho, u = _macros(f, F)
    if model == "cascaded":
        k = _forward(_forward(_grid(f), u[0], 0), u[1], 1)
        tr, df = k[2, 0] + k[0, 2], k[2, 0] - k[0, 2]
        tr = tr + om[0] * (2 / 3 * rho - tr)
        df = df - om[1] * df
        rows = [[rho, 0.5 * F[1] + 0 * rho, 0.5 * (tr - df)],
                [0.5 * F[0] + 0 * rho, (1 - om[2]) * k[1, 1], (1 - om[4]) * k[1, 2]],
                [0.5 * (tr + df), (1 - om[3]) * k[2, 1], k[2, 2] + om[5] * (rho / 9 - k[2, 2])]]
        return _from_central(torch.stack([torch.stack(r) for r in rows]), u)
    neq = f - _equilibrium(model, rho, u)
    if model == "bgk":
        out = f - om[1] * neq
        return out + (1 - 0.5 * om[1]) * _source(u, F) if forced else out
    K = torch.tensor(_K, dtype=torch.float64, device=f.device)
    rates = torch.tensor([0.0, 0.0, 0.0] + [float(w) for w in om], dtype=torch.float64, device=f.device)
    B = K.T @ torch.diag(rates / (K * K).sum(1)) @ K
    out = f - torch.tensordot(B, neq, 1)
    if forced:
        S = _source(u, F)
        out = out + S - 0.5 * torch.tensordot(B, S, 1)
    return out


def _stream(f, edges, wall_u, rho0=1.0):
    wall = [e != P for e in edges]
    U = [w if e == MW else 0.0 for e, w in zip(edges, wall_u)]
    out = []
    for q, ((x, y), w) in enumerate(zip(_E, _W)):
        g = torch.roll(f[q], (y, x), (0, 1))
        back = f[_OPP[q]]
        row = 0 if (y == 1 and wall[2]) else (-1 if (y == -1 and wall[3]) else None)
        col = 0 if (x == 1 and wall[0]) else (-1 if (x == -1 and wall[1]) else None)
        if row is not None:
            g[row, :] = back[row, :] + 6 * w * rho0 * x * (U[2] if row == 0 else U[3])
        if col is not None:
            g[:, col] = back[:, col] + 6 * w * rho0 * y * (U[0] if col == 0 else U[1])
        if row is not None and col is not None:
            g[row, col] = back[row, col]
        out.append(g)
    return torch.stack(out)


def _flow_exact(rho, u, F, om, model, edges, wall_u, steps, forced):
    f = _equilibrium(model, rho, u)
    if forced:
        f = f - 0.5 * _source(u, F)
    rows = max(1, (1 << 22) // f.shape[2])  # collide in bands: bounded temporaries on large lattices
    for _ in range(steps):
        if f.shape[1] <= rows:
            f = _collide(model, f, F, om, forced)
        else:
            for y in range(0, f.shape[1], rows):
                Fb = [v[y:y + rows] if torch.is_tensor(v) else v for v in F]
                f[:, y:y + rows] = _collide(model, f[:, y:y + rows], Fb, om, forced)
        f = _stream(f, edges, wall_u)
    return f


def _macros3(f, F):
    rho = f.sum((0, 1, 2))
    j = [f[2].sum((0, 1)) - f[0].sum((0, 1)), f[:, 2].sum((0, 1)) - f[:, 0].sum((0, 1)),
         f[:, :, 2].sum((0, 1)) - f[:, :, 0].sum((0, 1))]
    return rho, torch.stack([(j[i] + 0.5 * F[i]) / rho for i in range(3)])


def _flow3_exact(rho, u, F, om, steps):
    m = [1.0, 0.0, 1 / 3]
    shape = tuple(rho.shape)

    def back(k, u):
        return _inverse(_inverse(_inverse(k, u[2], 2), u[1], 1), u[0], 0)

    k = torch.zeros((3, 3, 3) + shape, dtype=torch.float64, device=rho.device)
    for i in range(3):
        for j in range(3):
            for l in range(3):
                k[i, j, l] = rho * (m[i] * m[j] * m[l])
    k[1, 0, 0], k[0, 1, 0], k[0, 0, 1] = -0.5 * F[0], -0.5 * F[1], -0.5 * F[2]
    f = back(k, u)
    for _ in range(steps):
        rho, u = _macros3(f, F)
        k = _forward(_forward(_forward(f, u[0], 0), u[1], 1), u[2], 2)
        xx, yy, zz = k[2, 0, 0].clone(), k[0, 2, 0].clone(), k[0, 0, 2].clone()
        tr, d1, d2 = xx + yy + zz, xx - yy, xx - zz
        tr, d1, d2 = tr + om[0] * (rho - tr), d1 - om[1] * d1, d2 - om[1] * d2
        for i in range(3):
            for j in range(3):
                for l in range(3):
                    o = i + j + l
                    if o >= 2:
                        w = om[1] if o == 2 else om[o - 1]
                        k[i, j, l] += w * (rho * (m[i] * m[j] * m[l]) - k[i, j, l])
        k[2, 0, 0], k[0, 2, 0], k[0, 0, 2] = (tr + d1 + d2) / 3, (tr - 2 * d1 + d2) / 3, (tr + d1 - 2 * d2) / 3
        k[1, 0, 0], k[0, 1, 0], k[0, 0, 1] = 0.5 * F[0], 0.5 * F[1], 0.5 * F[2]
        k = back(k, u)
        for i in range(3):
            for j in range(3):
                for l in range(3):
                    f[i, j, l] = torch.roll(k[i, j, l], (l - 1, j - 1, i - 1), (0, 1, 2))
    return _macros3(f, F)


def exact(case, seed):
    if case["kind"] == "flow":
        rho, u, force, field, om = _flow_inputs(case, seed)
        forced = case["force"] != "none"
        F = [field[0] + force[0], field[1] + force[1]] if field is not None else list(force)
        f = _flow_exact(rho, u, F, om, case["model"], EDGES[case["edges"]], (0.0, 0.0, 0.0, LID), case["steps"], forced)
        return list(_macros(f, F)) + ([f] if case["populations"] else [])
    if case["kind"] == "flow3":
        rho, u, F, om = _flow3_inputs(case, seed)
        return [t.cpu().numpy() for t in _flow3_exact(rho, u, F, om, case["steps"])]
    if case["kind"] == "gradient":
        u0, force, target, omega = _gradient_inputs(case, seed)
        w = torch.tensor(omega, dtype=torch.float64, device="cuda", requires_grad=True)
        u0.requires_grad_()
        force.requires_grad_()

        def segment(f, force, w, n):
            for _ in range(n):
                f = _stream(_collide("cascaded", f, force, (1.0, w, w, 1.0, 1.0, 1.0), True), EDGES["periodic"], (0.0,) * 4)
            return f

        f = _equilibrium("cascaded", torch.ones_like(u0[0]), u0) - 0.5 * _source(u0, force)
        left = case["steps"]
        while left > 0:
            n = min(20, left)
            f = torch.utils.checkpoint.checkpoint(segment, f, force, w, n, use_reentrant=False)
            left -= n
        loss = 0.5 * (_macros(f, force)[1] - target).square().sum()
        return [loss.detach()] + list(torch.autograd.grad(loss, (u0, force, w)))
    out = []
    for i, (n, edges, _, om) in enumerate(_domains(case)):
        rho, u = _modes(seed + 1000 * i, (n, n), 0.04)
        f = _flow_exact(rho, u, [0.0, 0.0], om, "cascaded", EDGES[edges], (0.0, 0.0, 0.0, LID), case["steps"], False)
        out += list(_macros(f, [0.0, 0.0]))
    return out
