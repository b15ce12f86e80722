"""The work that users of this library have it do, as measurable cases.

A case is one call sequence through the public Python interface
(``binding.Solver``, ``binding.MLP``): a stretch of lattice Boltzmann updates
between two samples of a run, the sampling itself, a whole run from host
arrays, a stretch of updates with the learned closure, a few training steps,
the gathering of training data. Sizes are those of ``configs.py``,
``dipole.py``, ``closure.py``, ``bench.py`` and the tests, or generic odd ones.

``exact`` evaluates the same method in 64 bits with plain torch operations
(Hermite sums as dense matrices, streaming by ``torch.roll``).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1505_06900_gb300 import binding as B
from paper_1505_06900_gb300 import workloads as W

STORAGES = {"f32": B.STORE_F32, "f16": B.STORE_F16, "bf16": B.STORE_BF16}
MODELS = {"rr": B.COLLIDE_RR, "reg2": B.COLLIDE_REG2, "bgk": B.COLLIDE_BGK}
CS2 = 1.0 / 3.0

# The most cell updates x directions of one drawn case: those of the largest
# listed one (D3Q27, 512^3, 20 updates).
MOST = 27 * 512 ** 3 * 20


def _step(name, q, shape, storage, walls, flow, mach, re, steps, model="rr"):
    return {"name": name, "kind": "step", "q": q, "nx": shape[0], "ny": shape[1], "nz": shape[2],
            "storage": storage, "walls": walls, "flow": flow, "mach": mach, "re": re,
            "steps": steps, "model": model}


def listed():
    return [
        # the smallest grid of configs.py between two samples (every = 50): launch latency
        _step("tgv2d_128", 9, (128, 128, 1), "f32", 0, "tgv", 0.05 * math.sqrt(3.0), 100.0, 50),
        # the double shear layer of configs.py between two samples: a 2-D store larger than L2
        _step("shear2d_2048", 9, (2048, 2048, 1), "f32", 0, "shear", 0.3, 1000.0, 50),
        # the dipole-wall benchmark of dipole.py at N = 500 between two samples (0.0025 time
        # units): odd rows, no-slip walls, a store that fits L2
        _step("dipole_n500", 9, (1001, 1001, 1), "f32", 3, "dipole", 0.0025 * math.sqrt(3.0),
              2500.0, 500),
        # the benchmark's headline workload and its default number of updates
        _step("tgv3d_512_f32", 27, (512, 512, 512), "f32", 0, "tgv", 0.1, 1600.0, 20),
        # its 16-bit form
        _step("tgv3d_512_f16", 27, (512, 512, 512), "f16", 0, "tgv", 0.1, 1600.0, 20),
        # the cheaper 3-D lattice on a box of no round size, the other 16-bit store
        _step("d3q19_ragged_bf16", 19, (250, 150, 101), "bf16", 0, "tgv", 0.1, 1600.0, 50),
        # a whole run from and to pinned host arrays (lb_run_host), as bench.py's end-to-end figure
        {"name": "host_256", "kind": "host", "q": 27, "nx": 256, "ny": 256, "nz": 256,
         "storage": "f32", "mach": 0.1, "re": 1600.0, "steps": 50},
        # one sample of a run (every 50 updates) after an odd number of updates: all fields,
        # the FP64 diagnostics, the enstrophy
        {"name": "sample_256", "kind": "sample", "q": 27, "nx": 256, "ny": 256, "nz": 256,
         "storage": "f32", "mach": 0.1, "re": 1600.0, "parity": 1},
        # the learned closure at the benchmark's coarse size
        {"name": "closure_256", "kind": "closure", "nx": 256, "ny": 256, "nz": 256, "mach": 0.3,
         "re": 1600.0, "steps": 10},
        # and at the coarse size of closure.py's default run
        {"name": "closure_64", "kind": "closure", "nx": 64, "ny": 64, "nz": 64, "mach": 0.3,
         "re": 1600.0, "steps": 20},
        # eight Adam steps at the recipe's batch, then the parameters
        {"name": "train_8192", "kind": "train", "batch": 8192, "steps": 8, "lr": 2e-3},
        # one snapshot of closure.py's data generation (fine 128^3) with the a-priori check
        {"name": "dataset_128", "kind": "dataset", "nx": 128, "ny": 128, "nz": 128, "mach": 0.3,
         "re": 1600.0},
    ]


def _size(rng, lo, hi):
    """A size between lo and hi, even over the logarithm: one half as it falls (odd ones among
    them), one half a multiple of 16, 64 or 128 where that fits."""
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    if rng.random() < 0.5:
        m = rng.choice([16, 64, 128])
        if n >= m:
            n = n // m * m
    return max(lo, min(hi, n))


def draw(rng):
    kind = rng.choices(["step", "host", "sample", "closure", "train", "dataset"],
                       [12, 1, 2, 2, 2, 1])[0]
    if kind == "train":
        return {"kind": kind, "batch": _size(rng, 100, 65536), "steps": rng.randint(1, 8),
                "lr": 2e-3}
    if kind == "closure":
        n = _size(rng, 16, 256)
        steps = max(1, min(40, int(256 ** 3 * 10 / n ** 3)))
        return {"kind": kind, "nx": n, "ny": _size(rng, max(8, n // 2), n),
                "nz": _size(rng, max(8, n // 2), n), "mach": 0.3, "re": 1600.0,
                "steps": rng.randint(max(1, steps // 4), steps)}
    if kind == "dataset":
        n = 2 * rng.randint(12, 80)
        return {"kind": kind, "nx": n, "ny": n, "nz": n, "mach": 0.3, "re": 1600.0}
    q = rng.choice([9, 9, 19, 27, 27])
    storage = rng.choice(["f32", "f32", "f16", "bf16"])
    if q == 9:
        nx, ny, nz = _size(rng, 64, 4096), _size(rng, 64, 4096), 1
    else:
        n = _size(rng, 24, 400)
        nx, ny, nz = n, _size(rng, max(16, n // 3), n), _size(rng, max(16, n // 3), n)
        if rng.random() < 0.4:  # a flat or long box of the same number of cells
            nx, nz = min(2 * nx, 640), max(5, nz // 2)
    base = {"q": q, "nx": nx, "ny": ny, "nz": nz, "storage": storage}
    if kind == "sample":
        return {"kind": kind, **base, "mach": 0.1, "re": 1600.0, "parity": rng.randint(0, 1)}
    most = max(1, min(200, MOST // (2 * q * nx * ny * nz)))
    steps = min(most, int(round(math.exp(rng.uniform(0.0, math.log(200.0))))))
    if kind == "host":
        return {"kind": kind, **base, "mach": 0.1, "re": 1600.0, "steps": steps}
    walls = rng.choice([0, 0, 0, 1, 2, 3] if q == 9 else [0, 0, 0, 0, 2, 7])
    flow = "shear" if q == 9 and not walls and rng.random() < 0.5 else "tgv"
    return {"kind": kind, **base, "walls": walls, "flow": flow,
            "mach": rng.choice([0.1, 0.3]) if q == 9 else 0.1,
            "re": 1000.0 if q == 9 else 1600.0, "steps": steps,
            "model": rng.choices(["rr", "reg2", "bgk"], [6, 1, 1])[0]}


# ------------------------------------------------------------------ inputs --
def _tau(case):
    n = max(case["nx"], case["ny"]) if case.get("q") == 9 else case["nx"] / (2.0 * math.pi)
    if case.get("flow") == "dipole":
        n = (case["nx"] - 1) // 2  # half the box, as in dipole.py
    return 0.5 + case["mach"] * math.sqrt(CS2) * n / case["re"] / CS2


def _fields64(case, seed):
    """rho [nz, ny, nx] and u [D, nz, ny, nx] (float64, on the GPU): the Taylor-Green vortex, the
    double shear layer or the dipole, at a phase (a place) and an amplitude of the seed."""
    rng = np.random.default_rng(seed)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    d = 2 if case.get("q") == 9 else 3
    u0 = case["mach"] * math.sqrt(CS2) * rng.uniform(0.95, 1.0)
    ph = rng.uniform(0.0, 2.0 * math.pi, 3)
    ar = lambda n: torch.arange(n, dtype=torch.float64, device="cuda")  # noqa: E731
    X = (2 * math.pi * (ar(nx) + 0.5) / nx + ph[0])[None, None, :]
    Y = (2 * math.pi * (ar(ny) + 0.5) / ny + ph[1])[None, :, None]
    flow = case.get("flow", "tgv")
    one = torch.ones((nz, ny, nx), dtype=torch.float64, device="cuda")
    if flow == "dipole":
        N = (nx - 1) // 2
        x, y = (-1.0 + ar(nx) / N)[None, None, :], (-1.0 + ar(ny) / N)[None, :, None]
        x, y = x - 0.2 * math.cos(ph[0]), y - 0.2 * math.sin(ph[0])
        we, r0 = W.DIPOLE_OMEGA_E, W.DIPOLE_R0
        e1 = torch.exp(-(x ** 2 + (y - 0.1) ** 2) / r0 ** 2)
        e2 = torch.exp(-(x ** 2 + (y + 0.1) ** 2) / r0 ** 2)
        ux = (-0.5 * we * (y - 0.1) * e1 + 0.5 * we * (y + 0.1) * e2) * u0
        uy = (0.5 * we * x * e1 - 0.5 * we * x * e2) * u0
        rho, u = one, torch.stack([ux * one, uy * one])
    elif flow == "shear":
        yy = torch.remainder((ar(ny) / ny + ph[1] / (2 * math.pi)), 1.0)[None, :, None]
        ux = torch.where(yy <= 0.5, u0 * torch.tanh(80.0 * (yy - 0.25)),
                         u0 * torch.tanh(80.0 * (0.75 - yy)))
        rho, u = one, torch.stack([ux * one, 0.05 * u0 * torch.sin(X) * one])
    elif d == 2:
        ux = u0 * (nx / max(nx, ny)) * torch.sin(X) * torch.cos(Y) * one
        uy = -u0 * (ny / max(nx, ny)) * torch.cos(X) * torch.sin(Y) * one
        rho = one - u0 * u0 / (4.0 * CS2) * (torch.cos(2 * X) + torch.cos(2 * Y))
        u = torch.stack([ux, uy])
    else:
        Z = (2 * math.pi * (ar(nz) + 0.5) / nz + ph[2])[:, None, None]
        ux = u0 * (nx / max(nx, ny)) * torch.sin(X) * torch.cos(Y) * torch.cos(Z) * one
        uy = -u0 * (ny / max(nx, ny)) * torch.cos(X) * torch.sin(Y) * torch.cos(Z) * one
        rho = one + u0 * u0 / (16.0 * CS2) * (torch.cos(2 * X) + torch.cos(2 * Y)) * (
            torch.cos(2 * Z) + 2.0)
        u = torch.stack([ux, uy, torch.zeros_like(ux)])
    for a, n in enumerate((nx, ny, nz)):  # at rest on the walls
        if (case.get("walls", 0) >> a) & 1:
            s = torch.sin(math.pi * ar(n) / (n - 1))
            s[0] = s[-1] = 0.0
            u = u * s.reshape([-1 if k == 2 - a else 1 for k in range(3)])
    return rho, u


def _fields(case, seed):
    return tuple(t.float().contiguous() for t in _fields64(case, seed))


def _params(seed):
    """Weights as they are some way into training, padded inputs and outputs at zero."""
    rng = np.random.default_rng(seed)
    W1 = rng.standard_normal((64, 288)) * math.sqrt(1.0 / 270)
    W1[:, 270:] = 0.0
    W2 = rng.standard_normal((64, 64)) * math.sqrt(1.0 / 64)
    W3 = rng.standard_normal((32, 64)) * math.sqrt(0.5 / 64)
    W3[17:] = 0.0
    b3 = 0.02 * rng.standard_normal(32)
    b3[17:] = 0.0
    return np.concatenate([W1.ravel(), 0.02 * rng.standard_normal(64), W2.ravel(),
                           0.02 * rng.standard_normal(64), W3.ravel(), b3]).astype(np.float32)


def _scaling(case, seed, out):
    """Mean and inverse spread of the moments of the flow, and the output scales."""
    rho, u = _fields64(case, seed)
    pi = _init_pi(rho, u, _tau(case))
    mom = torch.cat([(rho - 1.0)[None], u, pi]).reshape(10, -1)
    std = mom.std(1)
    std = torch.maximum(std, 1e-3 * std.max())
    return (mom.mean(1).cpu().numpy().astype(np.float32),
            (1.0 / std).cpu().numpy().astype(np.float32), np.full(17, out, np.float32))


def _solver(case, tau=None):
    return B.Solver(case.get("q", 27), (case["nx"], case["ny"], case["nz"]),
                    _tau(case) if tau is None else tau, storage=STORAGES[case.get("storage", "f32")],
                    collision=MODELS[case.get("model", "rr")], walls=case.get("walls", 0))


def _coarse(case):
    return {**case, "nx": case["nx"] // 2, "ny": case["ny"] // 2, "nz": case["nz"] // 2}


def prepare(case, seed):
    kind = case["kind"]
    if kind == "train":
        gen = torch.Generator(device="cuda").manual_seed(int(seed))
        n = case["batch"] * case["steps"]
        X = torch.randn((n, 288), device="cuda", generator=gen)
        X[:, 270:] = 0.0
        T = torch.randn((n, 32), device="cuda", generator=gen)
        T[:, 17:] = 0.0
        T[:, :17] = 0.5 * T[:, :17] + 0.5 * torch.sin(X[:, 130:147])
        X = X.to(torch.bfloat16)
        b = case["batch"]
        return {"case": case, "net": B.MLP(_params(seed)),
                "batches": [(X[k * b:(k + 1) * b], T[k * b:(k + 1) * b])
                            for k in range(case["steps"])]}
    if kind == "host":
        rho, u = _fields(case, seed)
        rho_h, u_h = rho.cpu().pin_memory(), u.cpu().pin_memory()
        return {"case": case, "solver": _solver(case), "rho": rho_h, "u": u_h,
                "rho_out": torch.empty_like(rho_h).pin_memory(),
                "u_out": torch.empty_like(u_h).pin_memory(), "diag": np.zeros(2 + u.shape[0])}
    s = _solver(case)
    s.init_fields(*_fields(case, seed))
    state = {"case": case, "solver": s}
    if kind == "sample":
        s.step(10 + case["parity"])
    elif kind == "closure":
        net = B.MLP(_params(seed))
        net.set_scaling(*_scaling(case, seed, 1e-5))
        s.set_closure(net, 8.0, 0.25)
        state["net"] = net
    elif kind == "dataset":
        net = B.MLP(_params(seed))
        c = _coarse(case)
        tau = 0.5 + (s.tau - 0.5) / 2.0
        net.set_scaling(*_scaling({**c, "re": case["re"]}, seed, 1e-4))
        state.update(net=net, a=_solver(c, tau), b=_solver(c, tau), scale=2.0 * tau / s.tau)
        s.step(24)
    torch.cuda.synchronize()
    return state


# --------------------------------------------------------------------- run --
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "train":
        net = state["net"]
        for X, T in state["batches"]:
            net.train_step(X, T, case["lr"], want_loss=False)
        return {"params": net.get_params()}
    s = state["solver"]
    if kind in ("step", "closure"):
        s.step(case["steps"])
        if case.get("walls"):  # fields: of a wall node's populations some are not in the flow
            return dict(zip(("rho", "u", "pi"), s.moments()))
        return {"populations": s.populations()}
    if kind == "host":
        s.run_host(state["rho"], state["u"], case["steps"], rho_out=state["rho_out"],
                   u_out=state["u_out"], diag_out=state["diag"])
        return {"rho": state["rho_out"], "u": state["u_out"], "diagnostics": state["diag"]}
    if kind == "sample":
        rho, u, pi = s.moments()
        return {"rho": rho, "u": u, "pi": pi, "diagnostics": s.diagnostics(),
                "enstrophy": s.enstrophy()}
    a, b, net = state["a"], state["b"], state["net"]
    a.coarsen_from(s, state["scale"])
    s.step(2)
    b.coarsen_from(s, state["scale"])
    X = a.closure_features(net)
    T = a.closure_step_targets(b, net)
    return {"features": X, "targets": T, "predictions": net.forward(X)}


# -------------------------------------------------------------------- work --
# FP32 operations of one cell update (moments, coefficients, synthesis)
FLOPS = {9: 160, 19: 330, 27: 450}
MLP_FLOPS = 2 * (288 * 64 + 64 * 64 + 64 * 32)


def work(case):
    """The state in and out and each output once; the arithmetic of every update."""
    kind = case["kind"]
    if kind == "train":
        rows = case["batch"] * case["steps"]
        return {"bytes": rows * (270 * 2 + 17 * 4) + 4 * 24736 * 7, "flops": 3 * rows * MLP_FLOPS}
    n = case["nx"] * case["ny"] * case["nz"]
    q = case.get("q", 27)
    d = 2 if q == 9 else 3
    size = 4 if case.get("storage", "f32") == "f32" else 2
    if kind == "step":
        out = 4 * (1 + d + (3 if d == 2 else 6)) if case.get("walls") else 4 * q
        return {"bytes": n * (2 * q * size + out), "flops": n * FLOPS[q] * case["steps"]}
    if kind == "closure":
        return {"bytes": n * q * (2 * 4 + 4), "flops": n * (FLOPS[q] + MLP_FLOPS) * case["steps"]}
    if kind == "host":  # fields in, the store out, fields out
        return {"bytes": n * (2 * 4 * (1 + d) + q * size), "flops": n * FLOPS[q] * case["steps"]}
    if kind == "sample":
        fields = 1 + d + (3 if d == 2 else 6)
        return {"bytes": n * (q * size + 4 * fields), "flops": n * 60}
    nc = n // 8  # fine state in and out, features, targets and predictions out
    return {"bytes": n * 27 * 4 * 2 + nc * (288 * 2 + 2 * 32 * 4),
            "flops": n * FLOPS[27] * 2 + nc * MLP_FLOPS}


# ------------------------------------------------------------------- exact --
def _vel(q):
    if q == 9:
        return [(i % 3 - 1, i // 3 - 1, 0) for i in range(9)]
    v = [(i % 3 - 1, i // 3 % 3 - 1, i // 9 - 1) for i in range(27)]
    return v if q == 27 else [c for c in v if abs(c[0]) + abs(c[1]) + abs(c[2]) < 3]


def _weights(q):
    if q == 19:
        return [(1 / 3, 1 / 18, 1 / 36)[sum(map(abs, c))] for c in _vel(19)]
    w = {0: 2 / 3, 1: 1 / 6, -1: 1 / 6}
    return [w[c[0]] * w[c[1]] * (w[c[2]] if q == 27 else 1.0) for c in _vel(q)]


def _t(a):
    return torch.tensor(a, dtype=torch.float64, device="cuda")


def _moment_matrix(q):
    """Rows: 1, x, y, z, xx, xy, xz, yy, yz, zz."""
    rows = []
    for p in ((), (0,), (1,), (2,), (0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2)):
        rows.append([math.prod(c[a] for a in p) for c in _vel(q)])
    return _t(rows)


POWERS = [(a, b, c) for a in range(3) for b in range(3) for c in range(3)]
HIGH = [(2, 1, 0), (2, 0, 1), (1, 2, 0), (1, 0, 2), (0, 1, 2), (0, 2, 1), (1, 1, 1), (2, 2, 0),
        (2, 0, 2), (0, 2, 2), (1, 1, 2), (1, 2, 1), (2, 1, 1), (2, 1, 2), (2, 2, 1), (1, 2, 2),
        (2, 2, 2)]


def _powers(q):
    return [p for p in POWERS if q != 9 or p[2] == 0]


def _synthesis(q):
    """Populations from coefficients: the Hermite sum w / norm H for D2Q9 and D3Q27 (POWERS
    order), the class expressions of the kept D3Q19 basis for D3Q19."""
    rows = []
    for c, w in zip(_vel(q), _weights(q)):
        if q != 19:
            g = [(1.0, 3.0 * x, 4.5 * (x * x - CS2)) for x in c]
            rows.append([w * g[0][a] * g[1][b] * g[2][e] for a, b, e in _powers(q)])
            continue
        # drho, jx, jy, jz, Axx, Axy, Axz, Ayy, Ayz, Azz, then A_abb in the order
        # xyy, xzz, xxy, yzz, xxz, yyz
        r = [0.0] * 16
        r[0] = 1.0
        diag = (4, 7, 9)
        for k in diag:
            r[k] -= 1.5
        axes = [a for a in range(3) if c[a]]
        third = {(0, 1): 10, (0, 2): 11, (1, 0): 12, (1, 2): 13, (2, 0): 14, (2, 1): 15}
        for a in axes:
            r[diag[a]] += 4.5
            r[1 + a] += 3.0 * c[a]
        if len(axes) == 1:
            a = axes[0]
            for b in range(3):
                if b != a:
                    r[third[a, b]] -= 9.0 * c[a]
        elif len(axes) == 2:
            a, b = axes
            r[{(0, 1): 5, (0, 2): 6, (1, 2): 8}[a, b]] += 9.0 * c[a] * c[b]
            r[third[a, b]] += 9.0 * c[a]
            r[third[b, a]] += 9.0 * c[b]
        rows.append([w * x for x in r])
    return _t(rows)


PAIRS = ((0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2))


def _coefficients(q, drho, u, j, pi, om1, model):
    """[K, n] for _synthesis; pi [6, n] in the order xx, xy, xz, yy, yz, zz."""
    rho = 1.0 + drho
    if q == 19:
        A = [om1 * pi[k] + j[a] * u[b] for k, (a, b) in enumerate(PAIRS)]
        P = {ab: om1 * pi[k] for k, ab in enumerate(PAIRS)}
        P.update({(b, a): v for (a, b), v in list(P.items())})
        diag = (A[0], A[3], A[5])
        third = [u[a] * diag[b] + 2.0 * u[b] * P[a, b]
                 for a, b in ((0, 1), (0, 2), (1, 0), (1, 2), (2, 0), (2, 1))]
        if model == "reg2":
            third = [torch.zeros_like(drho)] * 6
        return torch.stack([drho, j[0], j[1], j[2], *A, *third])
    one, zero = torch.ones_like(drho), torch.zeros_like(drho)
    p = [(one, u[a], u[a] * u[a]) for a in range(3)]
    d = [(zero, one, 2.0 * u[a]) for a in range(3)]
    h = (0.0, 0.0, 1.0)
    out = []
    for e in _powers(q):
        if e == (0, 0, 0):
            out.append(drho)
            continue
        if sum(e) == 1:
            out.append(j[e.index(1)])
            continue
        if model == "reg2" and sum(e) > 2:
            out.append(zero)
            continue
        v = [p[a][e[a]] for a in range(3)]
        dv = [d[a][e[a]] for a in range(3)]
        s = h[e[0]] * pi[0] * v[1] * v[2] + pi[1] * dv[0] * dv[1] * v[2]
        s = s + pi[2] * dv[0] * v[1] * dv[2] + h[e[1]] * pi[3] * v[0] * v[2]
        s = s + pi[4] * v[0] * dv[1] * dv[2] + h[e[2]] * pi[5] * v[0] * v[1]
        out.append(rho * v[0] * v[1] * v[2] + om1 * s)
    return torch.stack(out)


def _macro(M, f):
    m = M @ f
    j = m[1:4]
    u = j / (1.0 + m[0])
    pi = m[4:].clone()
    for k, (a, b) in enumerate(PAIRS):
        pi[k] -= j[a] * u[b] + (CS2 * m[0] if a == b else 0.0)
    return m[0], u, j, pi


def _init_pi(rho, u, tau):
    d = u.shape[0]
    axis = {0: 2, 1: 1, 2: 0}
    du = [[0.5 * (torch.roll(u[b], -1, axis[a]) - torch.roll(u[b], 1, axis[a]))
           if a < d and b < d else torch.zeros_like(rho) for b in range(3)] for a in range(3)]
    k = -2.0 * CS2 * rho * tau
    return torch.stack([k * 0.5 * (du[a][b] + du[b][a]) for a, b in PAIRS])


class _Exact:
    """The method in 64 bits: shifted logical populations f [Q, N]."""

    def __init__(self, case, seed, tau=None):
        self.q, self.model = case.get("q", 27), case.get("model", "rr")
        self.shape = (case["nz"], case["ny"], case["nx"])
        self.n = case["nx"] * case["ny"] * case["nz"]
        self.tau = _tau(case) if tau is None else tau
        self.om1 = 1.0 - 1.0 / self.tau
        self.M, self.S, self.w = _moment_matrix(self.q), _synthesis(self.q), _weights(self.q)
        self.vel = _vel(self.q)
        self.chunk = 1 << 22
        self._walls(case.get("walls", 0))
        if seed is None:
            return
        rho, u = (t.double() for t in _fields(case, seed))
        pi = _init_pi(rho, u, self.tau).reshape(6, -1)
        rho, u = rho.reshape(-1), u.reshape(u.shape[0], -1)
        if u.shape[0] == 2:
            u = torch.cat([u, torch.zeros_like(u[:1])])
        if self.edge is not None:
            u[:, self.edge] = 0.0
            pi[:, self.edge] = 0.0
        self.f = torch.empty((self.q, self.n), dtype=torch.float64, device="cuda")
        basis = "reg2" if self.model == "reg2" else "rr"
        for s in range(0, self.n, self.chunk):
            e = slice(s, s + self.chunk)
            self.f[:, e] = self.S @ _coefficients(self.q, rho[e] - 1.0, u[:, e],
                                                  rho[e] * u[:, e], pi[:, e], 1.0, basis)

    def _walls(self, walls):
        self.edge = None
        if not walls:
            return
        unknown = torch.zeros((self.q, *self.shape), dtype=torch.bool, device="cuda")
        for a in range(3):
            if (walls >> a) & 1:
                dim = 3 - a
                for i, c in enumerate(self.vel):
                    if c[a] == 1:
                        unknown[i].select(dim - 1, 0).fill_(True)
                    elif c[a] == -1:
                        unknown[i].select(dim - 1, self.shape[dim - 1] - 1).fill_(True)
        unknown = unknown.reshape(self.q, -1)
        self.edge = torch.nonzero(unknown.any(0))[:, 0]
        self.unknown = unknown[:, self.edge]

    def _edge_macro(self, f):
        """rho - 1 and Pi of the closed state of the wall nodes (at rest)."""
        unk = self.unknown
        opp = unk.flip(0)
        buried = unk & opp
        f = torch.where(unk & ~buried, f.flip(0), f)
        w = _t(self.w)[:, None]
        wb = (w * buried).sum(0)
        drho = torch.where(buried, torch.zeros_like(f), f).sum(0) / (1.0 - wb)
        f = torch.where(buried, w * drho, f)
        m = self.M @ f
        pi = m[4:].clone()
        for k, (a, b) in enumerate(PAIRS):
            if a == b:
                pi[k] -= CS2 * m[0]
        return m[0], torch.zeros_like(m[1:4]), pi

    def _edge_post(self, f):
        """Post-collision populations of the wall nodes."""
        drho, z, pi = self._edge_macro(f)
        return self.S @ _coefficients(self.q, drho, z, z, pi, self.om1, "rr")

    def collide(self, f, delta=None):
        drho, u, j, pi = _macro(self.M, f)
        if self.model == "bgk":
            eq = self.S @ _coefficients(self.q, drho, u, j, pi, 0.0, "rr")
            return f + (1.0 - self.om1) * (eq - f)
        c = _coefficients(self.q, drho, u, j, pi, self.om1, self.model)
        if delta is not None:
            for k, p in enumerate(HIGH):
                c[POWERS.index(p)] += self.om1 * delta[k]
        return self.S @ c

    def step(self, n, correction=None):
        for _ in range(n):
            delta = correction(self) if correction is not None else None
            edge = None
            if self.edge is not None:
                old = self.f[:, self.edge]
                edge = self._edge_post(old)
            for s in range(0, self.n, self.chunk):
                e = slice(s, s + self.chunk)
                self.f[:, e] = self.collide(self.f[:, e], None if delta is None else delta[:, e])
            if edge is not None:
                self.f[:, self.edge] = edge
            f = self.f.reshape(self.q, *self.shape)
            for i, (cx, cy, cz) in enumerate(self.vel):
                if cx or cy or cz:
                    f[i] = torch.roll(f[i], (cz, cy, cx), (0, 1, 2))

    def macro(self):
        parts = [_macro(self.M, self.f[:, s:s + self.chunk])
                 for s in range(0, self.n, self.chunk)]
        out = [torch.cat([p[k] for p in parts], -1) for k in range(4)]
        if self.edge is not None:
            drho, z, pi = self._edge_macro(self.f[:, self.edge])
            for v, edge in zip(out, (drho, z, z, pi)):
                v[..., self.edge] = edge
        return out

    def moment_field(self):
        drho, u, _, pi = self.macro()
        return torch.cat([drho[None], u, pi])


def _features(mom, shape, scaling):
    """Standardised features [10, 27 neighbours] of every cell, as [N, 270]."""
    mean, inv, _ = (_t(np.asarray(v, np.float64)) for v in scaling)
    z = ((mom - mean[:, None]) * inv[:, None]).reshape(10, *shape)
    cols = []
    for dz in (-1, 0, 1):
        for dy in (-1, 0, 1):
            for dx in (-1, 0, 1):
                cols.append(torch.roll(z, (-dz, -dy, -dx), (1, 2, 3)).reshape(10, -1).T)
    return torch.cat(cols, 1)


def _network(params):
    p = _t(np.asarray(params, np.float64))
    out, o = [], 0
    for shape in ((64, 288), (64,), (64, 64), (64,), (32, 64), (32,)):
        k = math.prod(shape)
        out.append(p[o:o + k].reshape(shape).clone())
        o += k
    return out


def _forward(net, X):
    W1, b1, W2, b2, W3, b3 = net
    h1 = torch.tanh(X @ W1[:, :X.shape[1]].T + b1)
    h2 = torch.tanh(h1 @ W2.T + b2)
    return h2 @ W3.T + b3, h1, h2


def _exact_train(case, seed):
    st = prepare(case, seed)
    net = _network(_params(seed))
    m = [torch.zeros_like(p) for p in net]
    v = [torch.zeros_like(p) for p in net]
    for t, (X, T) in enumerate(st["batches"], 1):
        X, T = X.double(), T.double()
        Y, h1, h2 = _forward(net, X)
        dy = torch.zeros_like(Y)
        dy[:, :17] = 2.0 * (Y - T)[:, :17] / (X.shape[0] * 17)
        d2 = (dy @ net[4]) * (1.0 - h2 * h2)
        d1 = (d2 @ net[2]) * (1.0 - h1 * h1)
        grads = [d1.T @ X, d1.sum(0), d2.T @ h1, d2.sum(0), dy.T @ h2, dy.sum(0)]
        for k, g in enumerate(grads):
            m[k] = 0.9 * m[k] + 0.1 * g
            v[k] = 0.999 * v[k] + 0.001 * g * g
            net[k] = net[k] - case["lr"] * (m[k] / (1 - 0.9 ** t)) / (
                torch.sqrt(v[k] / (1 - 0.999 ** t)) + 1e-8)
    return {"params": torch.cat([p.reshape(-1) for p in net])}


def _exact_closure(case, seed):
    scaling = _scaling(case, seed, 1e-5)
    net = _network(_params(seed))
    scale = _t(np.asarray(scaling[2], np.float64))

    def correction(e):
        mom = e.moment_field()
        mean, inv = (_t(np.asarray(v, np.float64))[:, None] for v in scaling[:2])
        z = ((mom - mean) * inv).reshape(10, *e.shape)
        pre = 0.0  # layer 1 summed over the 27 neighbours
        for nb in range(27):
            dx, dy, dz = nb % 3 - 1, nb // 3 % 3 - 1, nb // 9 - 1
            zz = torch.roll(z, (-dz, -dy, -dx), (1, 2, 3)).reshape(10, -1)
            pre = pre + net[0][:, 10 * nb:10 * nb + 10] @ zz
        h = torch.tanh(pre + net[1][:, None])
        h = torch.tanh(net[2] @ h + net[3][:, None])
        y = (net[4] @ h + net[5][:, None])[:17]
        y = torch.sign(y) * torch.clamp(y.abs() - 0.25, min=0.0)
        return y * scale[:, None]

    e = _Exact(case, seed)
    e.step(case["steps"], correction)
    return {"populations": e.f.reshape(27, *e.shape)}


def _exact_dataset(case, seed):
    fine = _Exact(case, seed)
    c = _coarse(case)
    tau = 0.5 + (fine.tau - 0.5) / 2.0
    scale = 2.0 * tau / fine.tau
    scaling = _scaling({**c, "re": case["re"]}, seed, 1e-4)

    def coarse():
        e = _Exact(c, None, tau)
        nz, ny, nx = e.shape
        f = fine.f.reshape(27, nz, 2, ny, 2, nx, 2).mean((2, 4, 6)).reshape(27, -1)
        drho, u, j, pi = _macro(e.M, f)
        eq = e.S @ _coefficients(27, drho, u, j, pi, 0.0, "rr")
        e.f = eq + scale * (f - eq)
        return e

    fine.step(24)
    a = coarse()
    fine.step(2)
    b = coarse()
    X = torch.zeros((a.n, 288), dtype=torch.float64, device="cuda")
    X[:, :270] = _features(a.moment_field(), a.shape, scaling)
    P = b.f.reshape(27, *b.shape).clone()
    for i, (cx, cy, cz) in enumerate(a.vel):
        P[i] = torch.roll(P[i], (-cz, -cy, -cx), (0, 1, 2))
    r = P.reshape(27, -1) - a.collide(a.f)
    H = _t([[math.prod((1.0, x, x * x - CS2)[k] for x, k in zip(v, p)) for v in a.vel]
            for p in HIGH])
    T = torch.zeros((a.n, 32), dtype=torch.float64, device="cuda")
    T[:, :17] = ((H @ r) / a.om1 / _t(np.asarray(scaling[2], np.float64))[:, None]).T
    return {"features": X, "targets": T, "predictions": _forward(_network(_params(seed)), X)[0]}


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return _exact_train(case, seed)
    if kind == "closure":
        if case["nx"] * case["ny"] * case["nz"] * case["steps"] > 2e8:
            return None  # a minute in 64 bits
        return _exact_closure(case, seed)
    if kind == "dataset":
        return _exact_dataset(case, seed)
    cells = case["nx"] * case["ny"] * case["nz"]
    if cells * case.get("steps", 1) > 3e9:
        return None
    e = _Exact(case, seed)
    e.step(10 + case["parity"] if kind == "sample" else case["steps"])
    if kind == "step" and e.edge is None:
        return {"populations": e.f.reshape(e.q, *e.shape)}
    drho, u, j, pi = e.macro()
    d = 2 if e.q == 9 else 3
    u, j = u[:d], j[:d]
    diag = torch.stack([cells + drho.sum(), *j.sum(1), 0.5 * (j * u).sum()])
    rho = (1.0 + drho).reshape(e.shape)
    u = u.reshape(d, *e.shape)
    if kind == "host":
        return {"rho": rho, "u": u, "diagnostics": diag}
    pi = (pi[[0, 1, 3]] if d == 2 else pi).reshape(-1, *e.shape)
    if kind == "step":
        return {"rho": rho, "u": u, "pi": pi}
    axis = {0: 2, 1: 1, 2: 0}
    du = lambda b, a: 0.5 * (torch.roll(u[b], -1, axis[a]) - torch.roll(u[b], 1, axis[a]))  # noqa: E731
    ens = (du(1, 0) - du(0, 1)) ** 2
    if d == 3:
        ens = ens + (du(2, 1) - du(1, 2)) ** 2 + (du(0, 2) - du(2, 0)) ** 2
    return {"rho": rho, "u": u, "pi": pi, "diagnostics": diag, "enstrophy": 0.5 * ens.sum()}
