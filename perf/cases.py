"""The work a user of this library has it do, as cases that can be timed and checked.

listed() names the cases, draw() gives more of the same ranges, prepare() makes
what a program has in hand before the call (fields on the host, a handle with
its state), run() is one pass through the public entry points, work() the bytes
and operations of a pass, and exact() the same outputs from a plain torch FP64
form of the discrete model (no code of this repository in it).

Fields come back through Simulation.fields into a page-locked buffer and are
kept as torch tensors of the handle's storage type on the GPU, as a program
that goes on with them in torch holds them.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

DT = {"fp64": torch.float64, "fp32": torch.float32, "fp16": torch.float16, "bf16": torch.bfloat16}
# Lattice-unit parameters of the benchmark workloads (the library's defaults).
PARAMS = dict(
    rho_l=1.0, rho_g=0.1, nu=0.1, sigma=1e-3, W_phi=4.0, M_phi=0.1,
    beta_phi=0.25, beta_psi=0.25, beta_inter=0.75, W0=4.0, tau0=320.0,
    eps_s=0.05, k=0.15, D=0.1, Omega=0.55, g=1e-6, grad_eps=1e-3,
    grad_eps_at=1e-2, s_e=1.0, s_eps=1.0,
    thermal=0, Le=1.0, latent=1.0, theta0=-0.55, cp=10.0)
THERMAL = dict(thermal=1, Le=50.0, latent=1.0, theta0=-0.55, cp=10.0)
R_SEED = 6.0
STIR = 0.02            # largest velocity of the stirred melt (lattice units)
ENSEMBLE = "256x256*32,512x384*32,1024x512*32"


def listed():
    return [
        # a run watched from Python: one step, then the FP64 diagnostics (the
        # smallest call: launches and latency are all of it)
        dict(name="watch 128x128 fp32", kind="watch", nx=128, ny=128, steps=1),
        # the validation run of the model: one seed, one bubble, FP64
        dict(name="seed+bubble 128x128 fp64", kind="2d", nx=128, ny=128, precision="fp64",
             thermal=False, sides="periodic", seeds=1, bubbles=1, steps=100, call="step"),
        # one domain of moderate size (the differentiation workload's lattice)
        dict(name="growth 512x512 fp32", kind="2d", nx=512, ny=512, precision="fp32",
             thermal=False, sides="periodic", seeds=4, bubbles=8, steps=100, call="step"),
        # the paper's bubble between two dendrites: symmetric sides, a wall
        # below, far field above, temperature lattice, a width that is no
        # multiple of a tile
        dict(name="section-4 200x400 thermal", kind="2d", nx=200, ny=400, precision="fp32",
             thermal=True, sides="bounded", seeds=2, bubbles=1, steps=100, call="step"),
        # the throughput workload
        dict(name="growth 4096x4096 fp32", kind="2d", nx=4096, ny=4096, precision="fp32",
             thermal=False, sides="periodic", seeds=64, bubbles=128, steps=50, call="step"),
        # fields in, steps, fields out in one call, an odd lattice
        dict(name="run 1999x2111 fp32", kind="2d", nx=1999, ny=2111, precision="fp32",
             thermal=False, sides="periodic", seeds=16, bubbles=32, steps=50, call="run"),
        # the reduced-precision storage form at its workload's size
        dict(name="growth 8192x4096 fp16", kind="2d", nx=8192, ny=4096, precision="fp16",
             thermal=False, sides="periodic", seeds=1, bubbles=1, steps=40, call="step"),
        # temperature coupling on a ragged lattice
        dict(name="thermal 3001x1501 fp32", kind="2d", nx=3001, ny=1501, precision="fp32",
             thermal=True, sides="periodic", seeds=16, bubbles=32, steps=50, call="step"),
        # many independent domains of uneven sizes in one handle
        dict(name="ensemble 96 domains fp32", kind="ensemble", sizes=ENSEMBLE, steps=32),
        # forward and backward: an objective of the final state and its gradient
        dict(name="adjoint 512x512 fp32", kind="adjoint", nx=512, ny=512, seeds=4, bubbles=8,
             steps=100, every=25),
        # three dimensions: dendrites in a melt, and with flow and bubbles
        dict(name="melt 256^3 fp32", kind="melt3", nx=256, ny=256, nz=256, precision="fp32",
             thermal=False, seeds=64, steps=40),
        dict(name="two-phase 256^3 fp32", kind="flow3", nx=256, ny=256, nz=256, precision="fp32",
             thermal=False, seeds=32, bubbles=64, steps=20),
    ]


def _log_between(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["2d"] * 6 + ["watch", "adjoint", "ensemble", "melt3", "flow3"])
    if kind == "watch":
        return dict(kind=kind, nx=_log_between(rng, 64, 700), ny=_log_between(rng, 64, 700),
                    steps=rng.choice([1, 1, 2, 5]))
    if kind == "adjoint":
        nx, ny = _log_between(rng, 96, 640), _log_between(rng, 96, 400)
        return dict(kind=kind, nx=nx, ny=ny, seeds=rng.randint(1, 4), bubbles=rng.randint(1, 6),
                    steps=rng.randint(20, 100), every=rng.choice([10, 20, 25, 50]))
    if kind == "ensemble":
        sizes = ",".join("%dx%d*%d" % (_log_between(rng, 96, 1024), _log_between(rng, 96, 512),
                                       rng.randint(2, 32)) for _ in range(rng.randint(2, 3)))
        return dict(kind=kind, sizes=sizes, steps=rng.randint(8, 32))
    if kind in ("melt3", "flow3"):
        precision = rng.choice(["fp32"] * 4 + ["fp64"])
        hi = 224 if precision == "fp32" else 64
        nx, ny, nz = (_log_between(rng, 32, hi) for _ in range(3))
        thermal = rng.random() < 0.4
        c = dict(kind=kind, nx=nx, ny=ny, nz=nz, precision=precision, thermal=thermal,
                 seeds=rng.randint(1, 32), steps=rng.randint(5, 16))
        return dict(c, bubbles=rng.randint(1, 48)) if kind == "flow3" else c
    precision = rng.choice(["fp32", "fp32", "fp32", "fp16", "bf16", "fp64"])
    plain = precision in ("fp32", "fp64")
    sides = "bounded" if plain and rng.random() < 0.2 else "periodic"
    thermal = plain and (sides == "bounded" or rng.random() < 0.3)
    side = _log_between(rng, 96, 3600 if precision != "fp64" else 400)
    aspect = math.exp(rng.uniform(-0.6, 0.6))
    nx, ny = max(64, int(side * aspect)), max(64, int(side / aspect))
    if rng.random() < 0.5:
        nx -= nx % 16      # the other half of the widths are whatever they are
    few = max(1, min(64, nx * ny // 200000))
    steps = max(4, min(100, int((4e8 if precision != "fp64" else 4e6) / (nx * ny))))
    call = "run" if not thermal and sides == "periodic" and rng.random() < 0.25 else "step"
    return dict(kind="2d", nx=nx, ny=ny, precision=precision, thermal=thermal, sides=sides,
                seeds=2 if sides == "bounded" else few, bubbles=1 if sides == "bounded" else 2 * few,
                steps=steps, call=call)


# ---------------------------------------------------------------------------
# Initial fields: seeds and bubbles in a stirred melt (FP64, on the GPU).
# ---------------------------------------------------------------------------
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _axis(n):
    return torch.arange(n, dtype=torch.float64, device=_device())


def _offset(a, c, n, periodic):
    d = a - c
    return d - n * torch.round(d / n) if periodic else d


def _objects(case, rng):
    """Seeds (x, y) and bubbles (x, y, R) at random places, kept apart where they fit."""
    nx, ny = case["nx"], case["ny"]
    if case.get("sides") == "bounded":
        r = nx * rng.uniform(0.08, 0.12)
        return ([(0.0, 0.0), (nx - 1.0, 0.0)],
                [(nx / 2.0 - 0.5, ny * rng.uniform(0.25, 0.4), r)])
    seeds = [(nx * rng.random(), ny * rng.random()) for _ in range(case["seeds"])]
    bubbles = []
    top = max(9.0, min(40.0, min(nx, ny) / 8.0))
    for _ in range(200 * case["bubbles"]):
        if len(bubbles) == case["bubbles"]:
            break
        x, y, r = nx * rng.random(), ny * rng.random(), rng.uniform(8.0, top)

        def apart(qx, qy, gap):
            dx, dy = abs(x - qx) % nx, abs(y - qy) % ny
            return math.hypot(min(dx, nx - dx), min(dy, ny - dy)) >= gap
        if (all(apart(a, b, r + q + 8.0) for a, b, q in bubbles)
                and all(apart(a, b, r + R_SEED + 8.0) for a, b in seeds)):
            bubbles.append((x, y, r))
    return seeds, bubbles


def _fields2(case, seed):
    """phi, psi, C, vx, vy, p [6, ny, nx] and the grain angle of each site."""
    rng = random.Random(seed)
    nx, ny = case["nx"], case["ny"]
    per = case.get("sides", "periodic") == "periodic"
    seeds, bubbles = _objects(case, rng)
    x, y = _axis(nx)[None, :], _axis(ny)[:, None]
    psi = torch.full((ny, nx), -1.0, dtype=torch.float64, device=_device())
    phi = torch.ones_like(psi)
    near = torch.full_like(psi, 1e30)
    angle = torch.zeros_like(psi)
    r_s = R_SEED if per else 10.0
    for sx, sy in seeds:
        th = rng.uniform(0.0, math.pi / 2)
        r = torch.sqrt(_offset(x, sx, nx, per) ** 2 + _offset(y, sy, ny, per) ** 2)
        psi = torch.maximum(psi, torch.tanh(math.sqrt(0.5) * (r_s - r) / PARAMS["W0"]))
        angle = torch.where(r < near, th, angle)
        near = torch.minimum(near, r)
    for bx, by, br in bubbles:
        r = torch.sqrt(_offset(x, bx, nx, per) ** 2 + _offset(y, by, ny, per) ** 2)
        phi = torch.minimum(phi, 0.5 + 0.5 * torch.tanh(math.sqrt(0.5) * (r - br) / (2 * PARAMS["W_phi"])))
    C = phi * (1.0 - (1.0 - PARAMS["k"]) * 0.5 * (1.0 + psi))
    # cells of a divergence-free flow, at rest in the solid
    kx, ky = (2 if per else 1) * math.pi / nx, (2 if per else 1) * math.pi / ny
    px, py = (rng.uniform(0, 6.28), rng.uniform(0, 6.28)) if per else (0.0, 0.0)
    a = STIR / max(kx, ky)
    fluid = 0.5 * (1.0 - psi)
    sx, cx = torch.sin(kx * (x + 0.5) + px), torch.cos(kx * (x + 0.5) + px)
    sy, cy = torch.sin(ky * (y + 0.5) + py), torch.cos(ky * (y + 0.5) + py)
    return torch.stack([phi, psi, C, a * ky * sx * cy * fluid, -a * kx * cx * sy * fluid,
                        torch.zeros_like(phi)]), angle


def _fields3(case, seed):
    """phi, psi, C, vx, vy, vz, p [7, nz, ny, nx]."""
    rng = random.Random(seed)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    x, y, z = _axis(nx)[None, None, :], _axis(ny)[None, :, None], _axis(nz)[:, None, None]

    def dist(c):
        return torch.sqrt(_offset(x, c[0], nx, True) ** 2 + _offset(y, c[1], ny, True) ** 2
                          + _offset(z, c[2], nz, True) ** 2)
    psi = torch.full((nz, ny, nx), -1.0, dtype=torch.float64, device=_device())
    phi = torch.ones_like(psi)
    for _ in range(case["seeds"]):
        c = [n * rng.random() for n in (nx, ny, nz)]
        psi = torch.maximum(psi, torch.tanh(math.sqrt(0.5) * (8.0 - dist(c)) / PARAMS["W0"]))
    for _ in range(case.get("bubbles", 0)):
        c, r = [n * rng.random() for n in (nx, ny, nz)], rng.uniform(6.0, 14.0)
        phi = torch.minimum(phi, 0.5 + 0.5 * torch.tanh(math.sqrt(0.5) * (dist(c) - r) / (2 * PARAMS["W_phi"])))
    C = phi * (1.0 - (1.0 - PARAMS["k"]) * 0.5 * (1.0 + psi))
    fluid = 0.5 * (1.0 - psi)
    tx, ty, tz = 2 * math.pi * x / nx, 2 * math.pi * y / ny, 2 * math.pi * z / nz
    p1, p2 = rng.uniform(0, 6.28), rng.uniform(0, 6.28)
    a = STIR if case["kind"] == "flow3" else 0.0
    one = torch.ones_like(phi)
    return torch.stack([phi, psi, C, a * torch.sin(ty + p1) * fluid, a * torch.sin(tz + p2) * fluid,
                        a * torch.cos(tx + p1) * fluid * one, torch.zeros_like(phi)])


def _params(case):
    return dict(PARAMS, **(THERMAL if case.get("thermal") else {}))


def _names2(case):
    return ["phi", "psi", "C", "U", "vx", "vy"] + (["theta"] if case.get("thermal") else [])


def _host(shape):
    return torch.empty(shape, dtype=torch.float64, pin_memory=torch.cuda.is_available())


def _to_host(t):
    out = _host(tuple(t.shape))
    out.copy_(t)
    return out


def _buffers(state, shape):
    """Where the fields of a pass go: page-locked memory, the same on the GPU, and the result."""
    state["out"] = _host(shape)
    state["raw"] = torch.empty(shape, dtype=torch.float64, device=_device())
    state["dev"] = torch.empty(shape, dtype=DT[state["case"].get("precision", "fp32")], device=_device())
    return state


def _to_device(state):
    state["raw"].copy_(state["out"], non_blocking=True)
    return state["dev"].copy_(state["raw"])


def _domains(case):
    """(nx, ny, eps_s) of every domain of an ensemble, and the seed of its fields."""
    out = []
    for part in case["sizes"].split(","):
        size, count = part.split("*")
        nx, ny = (int(v) for v in size.split("x"))
        out += [(nx, ny, 0.02 + 0.05 * ((7 * i) % 32) / 32.0) for i in range(int(count))]
    return out


def _domain_case(nx, ny, i):
    return dict(kind="2d", nx=nx, ny=ny, seeds=1 + i % 4, bubbles=1 + i % 6, sides="periodic")


# ---------------------------------------------------------------------------
def prepare(case, seed):
    from paper_2407_01651_gb300 import pf

    kind = case["kind"]
    if kind in ("melt3", "flow3"):
        shape = (case["nx"], case["ny"], case["nz"])
        f = _to_host(_fields3(case, seed))
        cls = pf.Simulation3F if kind == "flow3" else pf.Simulation3D
        sim = cls(shape, _params(case), case["precision"])
        if kind == "flow3":
            sim.set_fields_stack(f.numpy())
        else:
            sim.set_fields(f[1].numpy(), f[2].numpy())
        return _buffers(dict(case=case, sim=sim), (sim.field_planes,) + tuple(f.shape[1:]))
    if kind == "ensemble":
        doms = _domains(case)
        sim = pf.Simulation(doms, PARAMS, "fp32")
        for i, (nx, ny, _) in enumerate(doms):
            f, _ = _fields2(_domain_case(nx, ny, i), seed + 1000 * i)
            sim.set_fields_stack(i, _to_host(f).numpy())
        sites = sum(a * b for a, b, _ in doms)
        fields = [torch.empty(sites, device=_device()) for _ in range(5)]
        return _buffers(dict(case=case, sim=sim, doms=doms, fields=fields), (5 * sites,))
    f, angle = _fields2(dict(case, seeds=1, bubbles=1) if kind == "watch" else case, seed)
    f = _to_host(f)
    sim = pf.Simulation([(case["nx"], case["ny"])], _params(case), case.get("precision", "fp32"))
    if case.get("sides") == "bounded":
        sim.set_boundaries(0, pf.BC_SYMMETRIC, pf.BC_SYMMETRIC, pf.BC_WALL, pf.BC_FARFIELD)
    state = dict(case=case, sim=sim, f=f)
    if kind in ("watch", "adjoint") or case.get("call") == "run":
        sim.set_fields_stack(0, f.numpy())
    else:
        state["f"] = None
        sim.set_fields_stack(0, f.numpy(), angle.cpu().numpy() if _grains(case) else None)
    if kind == "2d":
        state["names"] = _names2(case)
        _buffers(state, (len(state["names"]), case["ny"], case["nx"]))
    return state


def _grains(case):
    """Small lattices take an orientation per grain, large ones the lattice's."""
    return case["kind"] == "2d" and case["call"] == "step" and case["nx"] * case["ny"] <= 1 << 20


def run(state):
    case, sim = state["case"], state["sim"]
    kind = case["kind"]
    if kind == "watch":
        sim.step(case["steps"])
        return sim.reduce(0)
    if kind == "adjoint":
        sim.set_fields_stack(0, state["f"].numpy())
        J, g = sim.adjoint_step(case["steps"], 1.0, 1.0, case["every"])
        return {"J": np.float32(J), "grad": np.asarray(g, dtype=np.float32)}
    out = state["out"]
    if kind == "ensemble":
        sim.step(case["steps"])
        flat, at = out.numpy(), 0
        for i, (nx, ny, _) in enumerate(state["doms"]):
            sim.fields(i, ("phi", "psi", "C", "vx", "vy"), out=flat[at:at + 5 * nx * ny])
            at += 5 * nx * ny
        parts = torch.split(_to_device(state), [5 * nx * ny for nx, ny, _ in state["doms"]])
        for q in range(5):
            torch.cat([p.view(5, -1)[q] for p in parts], out=state["fields"][q])
        return dict(zip(("phi", "psi", "C", "vx", "vy"), state["fields"]))
    if kind in ("melt3", "flow3"):
        sim.step(case["steps"])
        names = list(sim.fields(out.numpy()))
    elif case["call"] == "run":
        names = state["names"]
        sim.run(state["f"].numpy(), case["steps"], names, out=out.numpy().reshape(-1))
    else:
        names = state["names"]
        sim.step(case["steps"])
        sim.fields(0, names, out=out.numpy().reshape(-1))
    order = _order(kind, case)     # the planes of the buffer
    dev = _to_device(state)
    keep = ("mu", "p")    # differences of nearly equal sums: diagnostics, not fields to go on with
    assert len(names) == len(order)
    return {n: dev[i] for i, n in enumerate(order) if n not in keep}


def _order(kind, case):
    th = ["theta"] if case.get("thermal") else []
    if kind == "melt3":
        return ["psi", "C", "U"] + th
    if kind == "flow3":
        return ["phi", "psi", "C", "U", "p", "vx", "vy", "vz", "mu"] + th
    return ["phi", "psi", "C", "U", "vx", "vy"] + th


def work(case):
    """Per site and step: the state the model carries from one step to the next,
    read once and written once.  A conserved lattice whose even moments are
    slaved to its density needs that density and one value per opposite pair;
    so 2-D: f 9, phi + 4, g before 5, g after 1 + 2, C + 2, 1/a_s^2, v 2, Q, a
    grain byte (thermal: e 1 + 1 + 2 more); 3-D: g before 7, g after 1 + 3,
    C + 3, 1/a_s^2, Q, with flow f 19, phi + 6, v 3 (thermal: 1 + 1 + 3 more)."""
    kind = case["kind"]
    size = {"fp64": 8, "fp32": 4, "fp16": 2, "bf16": 2}[case.get("precision", "fp32")]
    wide = max(size, 4)     # lagged scalars are held in the type of the arithmetic
    th = bool(case.get("thermal"))
    if kind in ("melt3", "flow3"):
        sites = case["nx"] * case["ny"] * case["nz"]
        values = 17 + (19 + 7 + 3 if kind == "flow3" else 0) + (5 if th else 0)
        per, fields = 2 * values * size, len(_order(kind, case))
        flops = (1700 if kind == "flow3" else 400) + (150 if th else 0)
    else:
        sites = (sum(a * b for a, b, _ in _domains(case)) if kind == "ensemble"
                 else case["nx"] * case["ny"])
        per = 2 * ((9 + 4 + 5 + 3 + 2 + (4 if th else 0)) * size + 6 * wide) + 1
        fields = {"watch": 6 * wide / 8, "adjoint": 6, "ensemble": 5}.get(kind, len(_order(kind, case)))
        flops = 700 + (120 if th else 0)
    b = sites * (per * case["steps"] + 8 * fields)
    if case.get("call") == "run":
        b += sites * 48
    if kind == "adjoint":     # forward, then backward: the state and its adjoint in, the adjoint out
        b += sites * per * 1.5 * case["steps"]
        flops *= 4
    return {"bytes": float(b), "flops": float(sites * flops * case["steps"])}


# ---------------------------------------------------------------------------
# The discrete model in FP64 torch operations.  2-D fields are [batch, y, x].
# ---------------------------------------------------------------------------
C9 = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
W9 = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
W5 = [1 / 3] + [1 / 6] * 4
OPP = [0, 3, 4, 1, 2, 7, 8, 5, 6]
MIRX = [0, 3, 2, 1, 4, 6, 5, 8, 7]
M9 = np.array([[1] * 9, [-4, -1, -1, -1, -1, 2, 2, 2, 2], [4, -2, -2, -2, -2, 1, 1, 1, 1],
               [c[0] for c in C9], [0, -2, 0, 2, 0, 1, -1, -1, 1],
               [c[1] for c in C9], [0, 0, -2, 0, 2, 1, 1, -1, -1],
               [0, 1, -1, 1, -1, 0, 0, 0, 0], [0, 0, 0, 0, 0, 1, -1, 1, -1]], dtype=np.float64)


def _mix(A, fs):
    """sum_j A[i, j] fs[j] for every i, skipping zeros."""
    out = []
    for row in A:
        acc = None
        for a, f in zip(row, fs):
            if a != 0.0:
                acc = f * float(a) if acc is None else acc + f * float(a)
        out.append(acc if acc is not None else torch.zeros_like(fs[0]))
    return out


def _roll(a, cy, cx):
    return torch.roll(a, (cy, cx), dims=(-2, -1)) if (cx or cy) else a


def _pull(fs, i, bounded, w=None, far=None):
    cx, cy = C9[i]
    a = _roll(fs[i], cy, cx)
    if bounded and (cx or cy):
        a = a.clone()
        if cx:      # symmetric sides: the mirrored direction at the mirrored source
            xb = 0 if cx > 0 else -1
            a[..., :, xb] = _roll(fs[MIRX[i]], cy, 0)[..., :, xb]
        if cy:      # wall below, far field above
            yb = 0 if cy > 0 else -1
            own = fs[OPP[i]][..., yb, :]
            a[..., yb, :] = own if cy > 0 or far is None else 2 * w * far - own
    return a


def _pull_scalar(r, i, bounded):
    return _pull([r] * 9, i, bounded)


def _pad(X, bounded, kind):
    if not bounded:
        X = torch.cat([X[..., -1:, :], X, X[..., :1, :]], -2)
        return torch.cat([X[..., -1:], X, X[..., :1]], -1)
    flip = kind in ("vx", "vy")
    lo = -X[..., :1, :] if flip else X[..., :1, :]
    hi = X[..., -1:, :]
    hi = -hi if flip or kind == "U" else (-2.0 - hi if kind == "psi" else hi)
    X = torch.cat([lo, X, hi], -2)
    s = -1.0 if kind == "vx" else 1.0
    return torch.cat([s * X[..., :1], X, s * X[..., -1:]], -1)


def _grad_lap(X, bounded, kind):
    P = _pad(X, bounded, kind)
    ny, nx = X.shape[-2:]

    def at(cx, cy):
        return P[..., 1 + cy:1 + cy + ny, 1 + cx:1 + cx + nx]
    gx = gy = lap = 0.0
    for w, (cx, cy) in list(zip(W9, C9))[1:]:
        d = at(cx, cy) - X
        if cx:
            gx = gx + 3 * w * cx * d
        if cy:
            gy = gy + 3 * w * cy * d
        lap = lap + 6 * w * d
    return gx, gy, lap


def _derived(p):
    lam = p["D"] * p["tau0"] / ((47.0 / 75.0) * p["W0"] ** 2)
    mc = 1.0 - (1.0 - p["k"]) * p["Omega"]
    return lam, mc, -mc * p["Omega"] / (1.0 - (1.0 - p["k"]) * p["Omega"])


def _sources(p, phi, psi, C, theta=None):
    lam, mc, th = _derived(p)
    k = p["k"]
    U = (2 * C / (1 + k - (1 - k) * psi) - 1) / (1 - k)
    om = 1 - psi * psi
    Q = (4 * p["beta_psi"] * psi * om - 2 * p["beta_inter"] * (1 - phi) ** 2 * (1 + psi)
         - lam * om * om * ((th if theta is None else theta) + mc * U))
    return U, Q


def _start2(f6, p):
    phi, psi, C, vx, vy, pr = f6
    rho = p["rho_g"] + phi * (p["rho_l"] - p["rho_g"])
    v2 = vx * vx + vy * vy
    S = dict(f=[], h=[], gpre=[], gpost=[], s=[])
    for w, (cx, cy) in zip(W9, C9):
        cu = cx * vx + cy * vy
        S["f"].append(w * 3 * pr + rho * w * (3 * cu + 4.5 * cu * cu - 1.5 * v2))
        S["h"].append(w * phi * (1 + 3 * cu))
    S["f"][0] = S["f"][0] - 3 * pr
    for w, (cx, cy) in zip(W5, C9):
        S["gpre"].append(w * psi)
        S["gpost"].append(w * psi)
        S["s"].append(w * C * (1 + 3 * (cx * vx + cy * vy)))
    U, Q = _sources(p, phi, psi, C)
    S.update(r=torch.ones_like(phi), phi=phi, C=C, vx=vx, vy=vy, Q=Q)
    if p["thermal"]:
        theta = torch.full_like(phi, p["theta0"])
        H = p["cp"] * (theta - 0.5 * p["latent"] * (1 + psi))
        S["e"] = [rho * H - (2 / 3) * theta]
        S["e"] += [theta / 6 + 0.5 * rho * H * (cx * vx + cy * vy) for cx, cy in C9[1:5]]
        S["rhoHv"] = (rho * H * vx, rho * H * vy)
        _, Q = _sources(p, phi, psi, C, theta)
        S["Q"] = Q / (1 / p["Le"] + _derived(p)[1] * (1 + (1 - p["k"]) * U))
    # buoyancy reference: the mean density of each domain
    S["rho_bar"] = p["rho_g"] + phi.mean(dim=(-2, -1), keepdim=True) * (p["rho_l"] - p["rho_g"])
    return S


def _step2(S, p, ct, sn, eps, bounded):
    """One coupled step; returns the new state and the fields."""
    drho = p["rho_l"] - p["rho_g"]
    k, omk = p["k"], 1.0 - p["k"]
    f = [_pull(S["f"], i, bounded) for i in range(9)]
    h = [_pull(S["h"], i, bounded) for i in range(9)]
    s = [_pull(S["s"], i, bounded, W5[i], 1.0) for i in range(5)]
    g = []
    for i in range(5):
        post, r = _pull(S["gpost"], i, bounded, W5[i], -1.0), _pull_scalar(S["r"], i, bounded)
        g.append(S["gpre"][i] + r * (post - S["gpre"][i]))
    phi, psi, C, psio = sum(h), sum(g), sum(s), sum(S["gpre"])
    gpx, gpy, lphi = _grad_lap(phi, bounded, "phi")
    gsx, gsy, _ = _grad_lap(psi, bounded, "psi")
    xx, xy, _ = _grad_lap(S["vx"], bounded, "vx")
    yx, yy, _ = _grad_lap(S["vy"], bounded, "vy")
    vox, voy = S["vx"], S["vy"]
    rho = p["rho_g"] + phi * drho
    ge2 = p["grad_eps"] ** 2
    im = 1 / torch.sqrt(gpx * gpx + gpy * gpy + ge2)
    nfx, nfy = gpx * im, gpy * im
    mu = (2 * p["beta_phi"] * phi * (1 - phi) * (1 - 2 * phi)
          - 2 * p["beta_inter"] * (1 - phi) * (1 + psi) ** 2 - p["W_phi"] ** 2 * lphi)
    fs = 6 * p["sigma"] / (p["W_phi"] * math.sqrt(2 * p["beta_phi"]))
    kap = math.sqrt(2 * p["beta_phi"]) / p["W_phi"]
    ap = kap * phi * (1 - phi)
    Dx, Dy = p["M_phi"] * (gpx - ap * nfx), p["M_phi"] * (gpy - ap * nfy)
    div = (phi - S["phi"]) + vox * gpx + voy * gpy
    Fpx = fs * mu * gpx + drho * (div * vox + Dx * xx + Dy * xy)
    Fpy = fs * mu * gpy + drho * (div * voy + Dx * yx + Dy * yy) - (rho - S["rho_bar"]) * p["g"]
    jx = sum(c[0] * a for c, a in zip(C9, f) if c[0])
    jy = sum(c[1] * a for c, a in zip(C9, f) if c[1])
    vsx, vsy = (jx + 0.5 * Fpx) / rho, (jy + 0.5 * Fpy) / rho
    chi = 0.5 * (1 + psi)
    vx, vy = (1 - chi) * vsx, (1 - chi) * vsy
    Fx, Fy = Fpx - 2 * chi * rho * vsx, Fpy - 2 * chi * rho * vsy
    v2 = vx * vx + vy * vy
    grx, gry = drho * gpx, drho * gpy
    pr = 0.6 * (sum(f[1:]) + 0.5 * (vx * grx + vy * gry) - (2 / 3) * rho * v2)
    # flow and phase lattices: m* = m - S (m - m_eq) + (1 - S/2) M G
    s_nu = 1 / (3 * p["nu"] + 0.5)
    s_q = 8 * (2 - s_nu) / (8 - s_nu)
    s_phi = 1 / (3 * p["M_phi"] + 0.5)
    G1x = phi * vx - S["phi"] * vox + ap * nfx / 3
    G1y = phi * vy - S["phi"] * voy + ap * nfy / 3

    def collide(pops, eq, G, rate):
        R = np.diag(1 - np.array(rate))
        inv = M9.T / (M9 * M9).sum(1)
        A = inv @ R @ M9
        half = inv @ np.diag(1 - 0.5 * np.array(rate)) @ M9
        d = _mix(A, [a - b for a, b in zip(pops, eq)])
        gg = _mix(half, G)
        return [a + b + c for a, b, c in zip(eq, d, gg)]
    feq, Gf, heq, Gh = [], [], [], []
    for w, (cx, cy) in zip(W9, C9):
        cu, cF, cg = cx * vx + cy * vy, cx * Fx + cy * Fy, cx * grx + cy * gry
        feq.append(w * 3 * pr + rho * w * (3 * cu + 4.5 * cu * cu - 1.5 * v2))
        Gf.append(3 * w * (cF + cu * cg))
        heq.append(w * phi * (1 + 3 * cu))
        Gh.append(3 * w * (cx * G1x + cy * G1y))
    feq[0] = feq[0] - 3 * pr
    fn = collide(f, feq, Gf, [1, p["s_e"], p["s_eps"], 1, s_q, 1, s_q, s_nu, s_nu])
    hn = collide(h, heq, Gh, [1, 1, 1, s_phi, 1, s_phi, 1, 1, 1])
    # dendrite: anisotropy in the grain frame
    gxr, gyr = ct * gsx + sn * gsy, -sn * gsx + ct * gsy
    gm2 = gsx * gsx + gsy * gsy
    m = torch.sqrt(gm2 + ge2)
    nx_, ny_ = -gxr / m, -gyr / m
    n2, s4 = nx_ ** 2 + ny_ ** 2, nx_ ** 4 + ny_ ** 4
    a_s = 1 + eps * (4 * s4 - 3 * n2 * n2)
    iso = s4 + 0.75 * n2 * (1 - n2)
    pre = -16 * eps * a_s * m
    nxr, nyr = pre * nx_ * (nx_ ** 2 - iso), pre * ny_ * (ny_ ** 2 - iso)
    Nx, Ny = ct * nxr - sn * nyr, sn * nxr + ct * nyr
    as2 = a_s * a_s
    lam, mc, _ = _derived(p)
    theta = iF = None
    if p["thermal"]:
        e = [_pull(S["e"], i, bounded, W5[i], p["theta0"]) for i in range(5)]
        rhoH = sum(e)
        theta = rhoH / rho / p["cp"] + 0.5 * p["latent"] * (1 + psi)
    U, Q = _sources(p, phi, psi, C, theta)
    at = (-p["W0"] / (2 * math.sqrt(2)) * a_s * (1 + omk * U) * (psi - psio)
          / torch.sqrt(gm2 + p["grad_eps_at"] ** 2))
    if p["thermal"]:
        iF = 1 / (1 / p["Le"] + mc * (1 + omk * U))
        ux, uy, _ = _grad_lap(U, bounded, "U")
        Q = Q * iF + p["W0"] ** 2 * mc * omk * iF * iF * (ux * (as2 * gsx + Nx) + uy * (as2 * gsy + Ny))
    s1 = 1 / (3 * p["W0"] ** 2 / p["tau0"] * as2 * (1.0 if iF is None else iF) + 0.5)

    def q5(m0, Jx, Jy):
        return [m0 / 3, m0 / 6 + Jx / 2, m0 / 6 + Jy / 2, m0 / 6 - Jx / 2, m0 / 6 - Jy / 2]

    def flux(q, rate, ex, ey, Gx, Gy):
        ax, ay = q[1] - q[3], q[2] - q[4]
        return ax - rate * (ax - ex) + (1 - rate / 2) * Gx, ay - rate * (ay - ey) + (1 - rate / 2) * Gy
    gpost = q5(psi + (1.5 * Q - 0.5 * S["Q"]) / p["tau0"],
               *flux(g, s1, 0.0, 0.0, -Nx / (3 * as2), -Ny / (3 * as2)))
    # solute
    A = 1 + k - omk * psi
    q = 0.5 * (1 - psi)
    E = 2 * omk * p["D"] * q * C / (A * A)
    jv = p["D"] * q * C * kap * (1 - phi)
    ex = C * vx - E * gsx + omk * (at * gsx + jv * nfx)
    ey = C * vy - E * gsy + omk * (at * gsy + jv * nfy)
    sc = 1 / (3 * (2 * p["D"] * q / A) + 0.5)
    snew = q5(C, *flux(s, sc, ex, ey, C * vx - S["C"] * vox, C * vy - S["C"] * voy))
    N = dict(f=fn, h=hn, gpre=g, gpost=gpost, s=snew, r=1 / as2, phi=phi, C=C, vx=vx, vy=vy, Q=Q,
             rho_bar=S["rho_bar"])
    out = dict(phi=phi, psi=psi, C=C, U=U, vx=vx, vy=vy)
    if p["thermal"]:
        kT = p["Le"] * p["D"] * p["rho_l"] * p["cp"]
        sth = 1 / (3 * kT + 0.5)
        hx, hy = rhoH * vx, rhoH * vy
        rho_o = p["rho_g"] + S["phi"] * drho
        ox, oy = S["rhoHv"]
        Jx, Jy = flux(e, sth, hx, hy, hx - ox, hy - oy)
        N["e"] = [rhoH - 2 * theta / 3, theta / 6 + Jx / 2, theta / 6 + Jy / 2, theta / 6 - Jx / 2,
                  theta / 6 - Jy / 2]
        N["rhoHv"] = (hx, hy)
        out["theta"] = theta
    return N, out


def _exact2(case, f6, angle, eps, steps):
    p = _params(case)
    f6 = [a[None] if a.dim() == 2 else a for a in f6]
    S = _start2(f6, p)
    bounded = case.get("sides") == "bounded"
    ct, sn = (torch.cos(angle), torch.sin(angle)) if angle is not None else (1.0, 0.0)
    for _ in range(steps):
        S, out = _step2(S, p, ct, sn, eps, bounded)
    return S, out


# 3-D: D3Q19 for the flow and phase lattices, D3Q7 (w0 = 1/4, c_s^2 = 1/4) for the rest.
C19 = ([(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)]
       + [(1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1),
          (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)])
W19 = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
C7, W7 = C19[:7], [1 / 4] + [1 / 8] * 6


def _rows19(p):
    """sum over the moments with a rate s != 1 of (1 - s) M M^T / |M|^2."""
    s_nu = 1 / (3 * p["nu"] + 0.5)
    s_q = 8 * (2 - s_nu) / (8 - s_nu)
    rows = []
    for x, y, z in C19:
        c2 = x * x + y * y + z * z
        rows.append([19 * c2 - 30, (21 * c2 * c2 - 53 * c2 + 24) / 2, (5 * c2 - 9) * x,
                     (5 * c2 - 9) * y, (5 * c2 - 9) * z, 3 * x * x - c2, y * y - z * z, x * y,
                     y * z, x * z, (y * y - z * z) * x, (z * z - x * x) * y, (x * x - y * y) * z])
    M = np.array(rows).T
    rate = np.array([p["s_e"], p["s_eps"]] + [s_q] * 3 + [s_nu] * 5 + [s_q] * 3)
    return (M.T * ((1 - rate) / (M * M).sum(1))) @ M


def _roll3(a, c):
    return torch.roll(a, (c[2], c[1], c[0]), dims=(-3, -2, -1)) if any(c) else a


def _grad3(X):
    gx = gy = gz = lap = 0.0
    for w, c in list(zip(W19, C19))[1:]:
        d = _roll3(X, (-c[0], -c[1], -c[2])) - X
        gx = gx + 3 * w * c[0] * d if c[0] else gx
        gy = gy + 3 * w * c[1] * d if c[1] else gy
        gz = gz + 3 * w * c[2] * d if c[2] else gz
        lap = lap + 6 * w * d
    return (gx, gy, gz), lap


def _dot(c, v):
    t = [a * b for a, b in zip(c, v) if a]
    return sum(t) if t else 0.0


def _exact3(case, f7, steps):
    p = _params(case)
    flow = case["kind"] == "flow3"
    phi, psi, C = f7[0], f7[1], f7[2]
    v = [f7[3], f7[4], f7[5]]
    drho = p["rho_l"] - p["rho_g"]
    lam, mc, _ = _derived(p)
    k, omk = p["k"], 1 - p["k"]
    ge2 = p["grad_eps"] ** 2
    kap = math.sqrt(2 * p["beta_phi"]) / p["W_phi"]
    if not flow:
        phi = torch.ones_like(phi)
        v = [torch.zeros_like(phi) for _ in range(3)]
    rho_bar = p["rho_g"] + phi.mean() * drho
    A19 = torch.tensor(_rows19(p), dtype=torch.float64, device=phi.device)

    def density(ph):
        return p["rho_g"] + ph * drho if flow else torch.full_like(ph, p["rho_l"])

    def feq(pr, rho, v):
        v2 = _dot((1, 1, 1), [a * a for a in v])
        out = []
        for w, c in zip(W19, C19):
            cu = _dot(c, v)
            out.append(w * (3 * pr + rho * (3 * cu + 4.5 * cu * cu - 1.5 * v2)))
        out[0] = out[0] - 3 * pr
        return out
    if flow:
        F = torch.stack(feq(f7[6], density(phi), v))
        H = [w * phi * (1 + 3 * _dot(c, v)) for w, c in zip(W19, C19)]
    gpre = [w * psi for w in W7]
    gpost = [w * psi for w in W7]
    s = [w * C * (1 + 4 * _dot(c, v)) for w, c in zip(W7, C7)]
    r = torch.ones_like(phi)
    U, Qo = _sources(p, phi, psi, C)
    if p["thermal"]:
        theta = torch.full_like(phi, p["theta0"])
        rH = density(phi) * p["cp"] * (theta - 0.5 * p["latent"] * (1 + psi))
        e = [rH - 0.75 * theta] + [theta / 8 + 0.5 * rH * _dot(c, v) for c in C7[1:]]
        _, Qo = _sources(p, phi, psi, C, theta)
        Qo = Qo / (1 / p["Le"] + mc * (1 + omk * U))
    phio, Co, vo, jo = phi, C, v, None
    if p["thermal"]:
        jo = [rH * a for a in v]

    def q7(m0, J):
        out = [m0 / 4]
        for a in J:
            out += [m0 / 8 + a / 2, m0 / 8 - a / 2]
        return out
    for _ in range(steps):
        g = [gpre[i] + _roll3(r, C7[i]) * (_roll3(gpost[i], C7[i]) - gpre[i]) for i in range(7)]
        s = [_roll3(s[i], C7[i]) for i in range(7)]
        psi, psio, C = sum(g), sum(gpre), sum(s)
        gs, _ = _grad3(psi)
        nf = None
        if flow:
            h = [_roll3(H[i], C19[i]) for i in range(19)]
            for i in range(19):
                F[i] = _roll3(F[i], C19[i])
            phi = sum(h)
            gp, lphi = _grad3(phi)
            rho = density(phi)
            im = 1 / torch.sqrt(_dot((1, 1, 1), [a * a for a in gp]) + ge2)
            nf = [a * im for a in gp]
            mu = (2 * p["beta_phi"] * phi * (1 - phi) * (1 - 2 * phi)
                  - 2 * p["beta_inter"] * (1 - phi) * (1 + psi) ** 2 - p["W_phi"] ** 2 * lphi)
            fs = 6 * p["sigma"] / (p["W_phi"] * math.sqrt(2 * p["beta_phi"]))
            ap = kap * phi * (1 - phi)
            Dm = [p["M_phi"] * (a - ap * b) for a, b in zip(gp, nf)]
            div = (phi - phio) + sum(a * b for a, b in zip(vo, gp))
            Fp = []
            for q in range(3):
                dv, _ = _grad3(vo[q])
                Fp.append(fs * mu * gp[q] + drho * (div * vo[q] + sum(a * b for a, b in zip(Dm, dv))))
            Fp[1] = Fp[1] - (rho - rho_bar) * p["g"]
            j = [_dot([c[q] for c in C19], F) for q in range(3)]
            chi = 0.5 * (1 + psi)
            vs = [(a + 0.5 * b) / rho for a, b in zip(j, Fp)]
            v = [(1 - chi) * a for a in vs]
            Ft = [a - 2 * chi * rho * b for a, b in zip(Fp, vs)]
            v2 = sum(a * a for a in v)
            gr = [drho * a for a in gp]
            pr = 0.5 * (F[1:].sum(0) + 0.5 * sum(a * b for a, b in zip(v, gr)) - 0.5 * rho * v2)
            T = torch.stack(feq(pr, rho, v))
            for i, (w, c) in enumerate(zip(W19, C19)):
                if any(c):
                    T[i] += 1.5 * w * (_dot(c, Ft) + _dot(c, v) * _dot(c, gr))      # f_eq + G/2
            # f - (f_eq - G/2) = f - f_eq + G/2; G/2 = T - f_eq
            eq = torch.stack(feq(pr, rho, v))
            d = F - eq + (T - eq)
            del eq
            F = T + torch.matmul(A19, d.view(19, -1)).view_as(d)
            del T, d
            G1 = [phi * a - phio * b + ap * n / 3 for a, b, n in zip(v, vo, nf)]
            s_phi = 1 / (3 * p["M_phi"] + 0.5)
            flux = []
            for q in range(3):
                acc = 0.0
                for i, (w, c) in enumerate(zip(W19, C19)):
                    if c[q]:
                        acc = acc + c[q] * (h[i] - w * phi * (1 + 3 * _dot(c, v)) + 1.5 * w * _dot(c, G1))
                flux.append((1 - s_phi) * acc / 10)
            H = []
            for w, c in zip(W19, C19):
                H.append(w * phi * (1 + 3 * _dot(c, v)) + 1.5 * w * _dot(c, G1) + _dot(c, flux))
        gm2 = sum(a * a for a in gs)
        m = torch.sqrt(gm2 + ge2)
        n = [-a / m for a in gs]
        n2, s4 = sum(a * a for a in n), sum(a ** 4 for a in n)
        a_s = 1 + p["eps_s"] * (4 * s4 - 3 * n2 * n2)
        iso = s4 + 0.75 * n2 * (1 - n2)
        N = [-16 * p["eps_s"] * a_s * m * a * (a * a - iso) for a in n]
        as2 = a_s * a_s
        theta, iF = None, 1.0
        if p["thermal"]:
            e = [_roll3(e[i], C7[i]) for i in range(7)]
            rH = sum(e)
            theta = rH / (density(phi) * p["cp"]) + 0.5 * p["latent"] * (1 + psi)
        U, Q = _sources(p, phi, psi, C, theta)
        if p["thermal"]:
            gu, _ = _grad3(U)
            iF = 1 / (1 / p["Le"] + mc * (1 + omk * U))
            Q = Q * iF + p["W0"] ** 2 * iF * iF * mc * omk * sum(
                a * (as2 * b + c) for a, b, c in zip(gu, gs, N))
        at = (-p["W0"] / (2 * math.sqrt(2)) * a_s * (1 + omk * U) * (psi - psio)
              / torch.sqrt(gm2 + p["grad_eps_at"] ** 2))
        s1 = 1 / (4 * p["W0"] ** 2 / p["tau0"] * as2 * iF + 0.5)
        J = [(1 - s1) * (g[2 * q + 1] - g[2 * q + 2]) - (1 - s1 / 2) * N[q] / (4 * as2) for q in range(3)]
        gpre, gpost, r = g, q7(psi + (1.5 * Q - 0.5 * Qo) / p["tau0"], J), 1 / as2
        Qo = Q
        A = 1 + k - omk * psi
        qf = 0.5 * (1 - psi)
        E = 2 * omk * p["D"] * qf * C / (A * A)
        sc = 1 / (4 * (2 * p["D"] * qf / A) + 0.5)
        jv = p["D"] * qf * C * kap * (1 - phi)
        J = []
        for q in range(3):
            eq = C * v[q] - E * gs[q] + omk * (at * gs[q] + (jv * nf[q] if flow else 0.0))
            a = s[2 * q + 1] - s[2 * q + 2]
            J.append(a - sc * (a - eq) + (1 - sc / 2) * (C * v[q] - Co * vo[q]))
        s = q7(C, J)
        if p["thermal"]:
            sth = 1 / (4 * (p["Le"] * p["D"] * p["rho_l"] * p["cp"]) + 0.5)
            jn = [rH * a for a in v]
            E7 = [rH - 0.75 * theta]
            for q in range(3):
                a = e[2 * q + 1] - e[2 * q + 2]
                a = a - sth * (a - jn[q]) + (1 - sth / 2) * (jn[q] - jo[q])
                E7 += [theta / 8 + a / 2, theta / 8 - a / 2]
            e, jo = E7, jn
        phio, Co, vo = phi, C, v
    out = dict(phi=phi, psi=psi, C=C, U=U, vx=v[0], vy=v[1], vz=v[2], theta=theta)
    return {n: out[n] for n in _order(case["kind"], case) if n not in ("p", "mu")}


def _totals(out):
    """The diagnostics of one domain (FP64 totals over its sites)."""
    phi, psi, C, vx, vy = (out[n][0] for n in ("phi", "psi", "C", "vx", "vy"))
    ny, nx = phi.shape
    gas = 1 - phi
    t = dict(sum_phi=phi.sum(), sum_C=C.sum(), sum_hpsi=(0.5 * (1 + psi)).sum(), gas=gas.sum(),
             gas_x=(gas * _axis(nx)[None, :]).sum(), gas_y=(gas * _axis(ny)[:, None]).sum(),
             max_v=torch.sqrt(vx * vx + vy * vy).max())
    t = {n: float(v) for n, v in t.items()}
    return dict(t, p_in_sum=0.0, p_in_n=0.0, p_out_sum=0.0, p_out_n=0.0, nonfinite=0.0)


def exact(case, seed):
    kind = case["kind"]
    with torch.no_grad():
        if kind in ("melt3", "flow3"):
            return _exact3(case, list(_fields3(case, seed)), case["steps"])
        if kind == "ensemble":
            doms, parts = _domains(case), {}
            for size in sorted({d[:2] for d in doms}):
                at = [i for i, d in enumerate(doms) if d[:2] == size]
                f6 = torch.stack([_fields2(_domain_case(*size, i), seed + 1000 * i)[0] for i in at], 1)
                eps = torch.tensor([doms[i][2] for i in at], dtype=torch.float64,
                                   device=f6.device).view(-1, 1, 1)
                _, out = _exact2(case, list(f6), None, eps, case["steps"])
                for b, i in enumerate(at):
                    parts[i] = {n: out[n][b].reshape(-1) for n in ("phi", "psi", "C", "vx", "vy")}
            return {n: torch.cat([parts[i][n] for i in range(len(doms))])
                    for n in ("phi", "psi", "C", "vx", "vy")}
        if kind != "adjoint":
            f6, angle = _fields2(dict(case, seeds=1, bubbles=1) if kind == "watch" else case, seed)
            _, out = _exact2(case, list(f6), angle if _grains(case) else None, PARAMS["eps_s"], case["steps"])
            if kind == "watch":
                return _totals(out)
            return {n: out[n][0] for n in _order(kind, case)}
    return _exact_adjoint(case, seed)


def _exact_adjoint(case, seed):
    """J = mean h(psi_T) + y_c(T) / L_y and its gradient by reverse-mode torch."""
    from torch.utils.checkpoint import checkpoint

    f6, _ = _fields2(case, seed)
    th = [torch.tensor(PARAMS[n], dtype=torch.float64, device=f6.device, requires_grad=True)
          for n in ("eps_s", "Omega", "sigma")]
    p = dict(_params(case), Omega=th[1], sigma=th[2])
    S = _start2([a[None] for a in f6], p)
    keys = list(S)
    flat = []
    for n in keys:
        flat += S[n] if isinstance(S[n], list) else [S[n]]

    def one(eps, Om, sg, *vals):
        it, st = iter(vals), {}
        for n in keys:
            st[n] = [next(it) for _ in S[n]] if isinstance(S[n], list) else next(it)
        new, out = _step2(st, dict(p, Omega=Om, sigma=sg), 1.0, 0.0, eps, False)
        back = []
        for n in keys:
            back += new[n] if isinstance(new[n], list) else [new[n]]
        return tuple(back) + (out["phi"], out["psi"])
    for _ in range(case["steps"]):
        res = checkpoint(one, *th, *flat, use_reentrant=False)
        flat, phi, psi = list(res[:-2]), res[-2][0], res[-1][0]
    gas = 1 - phi
    yc = (gas * _axis(case["ny"])[:, None]).sum() / gas.sum()
    J = (0.5 * (1 + psi)).mean() + yc / case["ny"]
    grad = torch.autograd.grad(J, th)
    return {"J": J.detach(), "grad": torch.stack([g.detach() for g in grad])}
