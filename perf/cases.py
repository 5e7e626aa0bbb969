"""Performance cases: what a program that uses the solver has it do.

``listed()`` names the cases, ``draw(rng)`` makes more of the same ranges.  A case is run with
``run(prepare(case, seed))``: through ``binding.Grid`` (a whole solve of a pulse table, in order or
with the time axis split into segments, and the projection of a state that is on the device),
``binding.density_noalloc`` (the density of a map the caller holds) or ``serve.run`` (a stream of
requests).  ``work(case)`` is what one pass cannot do without, and ``exact(case, seed)`` the result
of the same steps in 64 bits, in plain torch.

Units: hbar = v_F = e = 1; momenta and energies in eV, time in hbar/eV.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_1607_03062_gb300 import binding as B
from paper_1607_03062_gb300 import serve

TWO_PI = 2.0 * math.pi
HBAR_EVS = 6.582119569e-16
HBAR_VF_EVM = HBAR_EVS * 1.093e6

# FLOPs of one time step of one spinor that no arrangement of the step does without: dt (p + A) (2),
# its square (3), the two trigonometric factors of it (at least 4), their products with dt P (2), and
# the 2x2 update with a real diagonal (4 multiplications and 8 multiply-adds: 20).
FLOPS_PER_STEP = 31
# A point's projection on u(p + A_out): the unit vector (6), c+ (8) and |c+|^2 (4).
FLOPS_PROJECT = 18
# The 64-bit result of more spinor-steps than this takes too long.
EXACT_MOST = 2.4e10


def _solve(name, nx, ny, extent, pulse, E0, omega, cycles, steps, precision="fp32_mixed",
           scheme="exact", valley=1, eps=0.0, kind="solve", **more):
    return {"name": name, "kind": kind, "nx": nx, "ny": ny, "extent_x": extent,
            "extent_y": extent, "pulse": pulse, "E0": E0, "omega": omega, "cycles": cycles,
            "eps": eps, "steps": steps, "precision": precision, "scheme": scheme,
            "valley": valley, **more}


def listed():
    return [
        # The smallest solve: the FP64 parity workload (64 x 64, 5-cycle sin^2 pulse), one point of
        # a parameter scan.
        _solve("sin2_64_fp64", 64, 64, 4.0, "sin2", 1.0, 1.55, 5.0, 2000, "fp64"),
        # The same workload as a scan runs it when the time of one small grid counts: FP32-mixed,
        # the time axis in as many segments as the library picks.
        _solve("sin2_64_segmented", 64, 64, 4.0, "sin2", 1.0, 1.55, 5.0, 2000, kind="segmented"),
        # The paper's laser pulse (Sec. IV) on the grid the command line solves it on.
        _solve("paper_256", 256, 256, 0.5, "paper", 7.19e-3, 0.041357, 5.5, 20000),
        # An odd grid in FP64: the 300 x 257 box that is cut into row bands, elliptical pulse.
        _solve("ragged_300x257_fp64", 300, 257, 4.0, "sin2", 1.5, 1.3, 4.0, 1700, "fp64", eps=0.3),
        # A grid whose rows are no multiple of anything, two-colour elliptical pulse.
        _solve("ragged_1000x750", 1000, 750, 6.0, "two_colour", 3.0, 1.55, 10.0, 20000, eps=0.5),
        # 1024 x 1024, Gaussian pulse, 3e4 steps.
        _solve("gauss_1024", 1024, 1024, 8.0, "gauss", 2.0, 1.55, 4.0, 30000),
        # The fourth-order Magnus steps, valley K-, elliptical pulse.
        _solve("magnus4_512", 512, 512, 6.0, "sin2", 2.0, 1.55, 5.0, 12000, scheme="magnus4",
               valley=-1, eps=0.5),
        # The sigma_x / sigma_y split steps.
        _solve("strang_512x384", 512, 384, 6.0, "sin2", 2.0, 1.55, 5.0, 12000,
               scheme="strang_xy", eps=0.3),
        # A batch of requests through the continuous-batching server, results with their maps.
        {"name": "serving_16", "kind": "serving", "requests": 16, "n_most": 1024,
         "steps_most": 12000, "chunk": 2000, "precision": "fp32_mixed", "scheme": "exact",
         "valley": 1},
        # The benchmark: 2048 x 2048, 20-cycle sin^2 pulse, 1e5 steps, one sample of the scan.
        _solve("lzs_2048", 2048, 2048, 10.0, "sin2", 2.5, 1.9, 20.0, 100000),
        # The projection of an FP64 state that is on the device, on the largest grid.
        _solve("project_4096_fp64", 4096, 4096, 12.0, "two_colour", 3.0, 1.55, 10.0, 64, "fp64",
               eps=0.5, kind="project"),
        # The density of an FP32-mixed map that the caller holds, on the largest grid.
        {"name": "density_4096", "kind": "density", "nx": 4096, "ny": 4096, "extent_x": 12.0,
         "extent_y": 12.0, "precision": "fp32_mixed"},
    ]


def _size(rng, least, most):
    """A grid edge: half of them a power of two, half any number, odd ones among them."""
    n = math.exp(rng.uniform(math.log(least), math.log(most)))
    if rng.random() < 0.5:
        n = 2 ** round(math.log2(n))
    return max(least, min(most, int(n)))


def _pulse(rng):
    kind = rng.choice(["sin2", "sin2", "gauss", "two_colour", "paper"])
    if kind == "paper":
        return {"pulse": "paper", "E0": 7.19e-3 * rng.uniform(0.5, 2.0), "omega": 0.041357,
                "cycles": 5.5, "eps": 0.0}, 0.5
    cycles = {"sin2": rng.uniform(3.0, 20.0), "gauss": rng.uniform(1.0, 4.0),
              "two_colour": rng.uniform(5.0, 10.0)}[kind]
    return {"pulse": kind, "E0": rng.uniform(0.2, 6.0), "omega": rng.uniform(0.5, 3.0),
            "cycles": cycles, "eps": rng.choice([0.0, rng.uniform(0.0, 1.0)])}, rng.uniform(4.0, 12.0)


def draw(rng):
    kind = rng.choice(["solve"] * 11 + ["segmented"] * 2 + ["serving"] * 2 + ["project"] * 3 +
                      ["density"] * 2)
    precision = rng.choice(["fp32_mixed", "fp32_mixed", "fp64"])
    if kind == "serving":
        return {"kind": kind, "requests": rng.randint(6, 24), "n_most": rng.choice([256, 512, 1024]),
                "steps_most": rng.randint(2000, 16000), "chunk": rng.choice([1000, 2000, 4000]),
                "precision": "fp32_mixed", "scheme": "exact", "valley": rng.choice([1, -1])}
    if kind == "density":
        return {"kind": kind, "nx": _size(rng, 64, 4096), "ny": _size(rng, 64, 4096),
                "extent_x": rng.uniform(4.0, 12.0), "extent_y": rng.uniform(4.0, 12.0),
                "precision": precision}
    pulse, extent = _pulse(rng)
    case = {"kind": kind, "extent_x": extent, "extent_y": extent * rng.uniform(0.5, 1.0), **pulse,
            "precision": precision, "scheme": rng.choice(["exact"] * 4 + ["strang_xy", "magnus4"]),
            "valley": rng.choice([1, -1])}
    if kind == "project":
        case.update(nx=_size(rng, 256, 4096), ny=_size(rng, 256, 4096), steps=64)
        return case
    # The step count resolves the largest phase dt |p + A| to theta, as a user picks it.
    theta = math.exp(rng.uniform(math.log(0.005), math.log(0.06)))
    reach = math.hypot(extent, case["extent_y"]) + 1.5 * case["E0"] / case["omega"]
    case["steps"] = min(200000, max(500, int(_duration(case) * reach / theta)))
    case["nx"] = _size(rng, 48, 2048 if kind == "solve" else 128)
    case["ny"] = max(16, _size(rng, 48, 2048 if kind == "solve" else 128))
    # No dearer than the largest listed case, in each precision and scheme.
    most = 1.2e9 if precision == "fp64" else 1.5e11
    while case["nx"] * case["ny"] * case["steps"] > most:
        if case["nx"] * case["ny"] > 48 * 48:
            case["nx"], case["ny"] = max(48, case["nx"] * 3 // 4), max(48, case["ny"] * 3 // 4)
        else:
            case["steps"] = case["steps"] * 3 // 4
    return case


# ------------------------------------------------------------------------------------------
# Inputs
# ------------------------------------------------------------------------------------------

def _duration(case):
    period = TWO_PI / case["omega"]
    return period * case["cycles"] * (6.0 if case["pulse"] == "gauss" else 1.0)


def _int_cos(a, b, w, ph):
    """The integral of cos(w t + ph) over [a, b]."""
    z = 0.5 * w * (b - a)
    return (b - a) * np.cos(0.5 * w * (a + b) + ph) * np.sinc(z / np.pi)


def _potential(case, t):
    """A(t), an array [len(t), 2]."""
    E0, w, T, eps = case["E0"], case["omega"], _duration(case), case["eps"]
    t = np.asarray(t, dtype=np.float64)
    if case["pulse"] == "paper":  # A_x = -int E0 envelope cos(w t): sin^2 rise, flat, cos^2 fall
        om = 7.85e12 * HBAR_EVS
        tr, tf = math.pi / (2.0 * om), T - math.pi / (2.0 * om)
        b = np.minimum(t, tr)
        acc = (0.5 * _int_cos(0.0, b, w, 0.0) - 0.25 * _int_cos(0.0, b, w + 2 * om, 0.0)
               - 0.25 * _int_cos(0.0, b, w - 2 * om, 0.0))
        acc = acc + np.where(t > tr, _int_cos(tr, np.clip(t, tr, tf), w, 0.0), 0.0)
        b = np.maximum(t, tf)
        acc = acc + (0.5 * _int_cos(tf, b, w, 0.0) + 0.25 * _int_cos(tf, b, w + 2 * om, -2 * om * tf)
                     + 0.25 * _int_cos(tf, b, w - 2 * om, 2 * om * tf))
        return np.stack([-E0 * acc, np.zeros_like(t)], axis=-1)
    if case["pulse"] == "gauss":
        tau = T / 6.0
        f = np.exp(-((t - 0.5 * T) / tau) ** 2)
    else:
        f = np.sin(math.pi * t / T) ** 2
    ax, ay = np.sin(w * t), np.cos(w * t)
    if case["pulse"] == "two_colour":
        ax = ax + 0.5 * np.sin(2 * w * t + math.pi / 3)
        ay = ay + 0.5 * np.cos(2 * w * t + math.pi / 3)
    return (E0 / w) * np.stack([f * ax, eps * f * ay], axis=-1)


def _seeded(case, seed):
    """The case with its field strength and frequency a little off, by the seed."""
    r = random.Random(seed)
    return {**case, "E0": case["E0"] * r.uniform(0.97, 1.03),
            "omega": case["omega"] * r.uniform(0.98, 1.02)}


def _table(case):
    """The pulse as a solve takes it: samples, dt, A_in, A_out."""
    n, dt, t0 = case["steps"], _duration(case) / case["steps"], 0.0
    if case["kind"] == "project":  # a few steps at the peak of the pulse
        dt, t0 = _duration(case) / 20000, 0.5 * _duration(case)
    k = np.arange(n)
    if case["scheme"] == "magnus4":
        s = math.sqrt(3.0) / 6.0
        a = np.concatenate([_potential(case, t0 + (k + 0.5 - s) * dt),
                            _potential(case, t0 + (k + 0.5 + s) * dt)], axis=-1)
    else:
        a = _potential(case, t0 + (k + 0.5) * dt)
    ends = _potential(case, np.array([t0, t0 + n * dt]))
    return np.ascontiguousarray(a), dt, ends[0].copy(), ends[1].copy()


def _box(case):
    return (-case["extent_x"], case["extent_x"]), (-case["extent_y"], case["extent_y"])


def _requests(case, seed):
    """The stream of a serving case: grids of 128 points an edge and up, elliptical 5-cycle pulses."""
    r = random.Random("%d requests" % seed)
    sizes = [m for m in (1024, 512, 256, 128) if m <= case["n_most"]]
    out = []
    for k in range(case["requests"]):
        n = sizes[k % len(sizes)]
        out.append({"nx": n, "ny": n, "extent_x": 8.0, "extent_y": 8.0, "pulse": "sin2",
                    "E0": r.uniform(0.5, 4.0), "omega": r.uniform(0.8, 2.5), "cycles": 5.0,
                    "eps": r.uniform(0.0, 1.0), "steps": r.randint(1000, case["steps_most"]),
                    "kind": "solve", "scheme": case["scheme"],
                    "precision": case["precision"], "valley": case["valley"]})
    return out


def prepare(case, seed):
    if case["kind"] == "density":
        g = torch.Generator(device="cuda").manual_seed(seed)
        dt = torch.float64 if case["precision"] == "fp64" else torch.float32
        # |c+|^2 lies in [0, 1] and is small at most momenta
        m = torch.rand(case["ny"], case["nx"], dtype=dt, device="cuda", generator=g) ** 4
        return {"case": case, "map": m, "stream": torch.cuda.current_stream().cuda_stream}
    if case["kind"] == "serving":
        reqs = []
        for c in _requests(case, seed):
            a, dt, a_in, a_out = _table(c)
            px, py = _box(c)
            reqs.append({"grid": {"nx": c["nx"], "ny": c["ny"], "px": px, "py": py},
                         "steps": c["steps"], "arrival_s": 0.0, "precision": c["precision"],
                         "table": (a, a_in, a_out, dt)})
        return {"case": case, "requests": reqs, "stream": torch.cuda.current_stream().cuda_stream}
    c = _seeded(case, seed)
    px, py = _box(c)
    grid = B.Grid(c["nx"], c["ny"], px, py, c["precision"], c["scheme"], c["valley"])
    table = _table(c)
    if case["kind"] == "project":
        grid.set_pulse(*table)
        grid.evolve(c["steps"])
    return {"case": case, "grid": grid, "table": table}


def run(state):
    case = state["case"]
    if case["kind"] == "density":
        px, py = _box(case)
        return {"density": B.density_noalloc(state["map"].data_ptr(), case["precision"], case["nx"],
                                             case["ny"], px, py, state["stream"])}
    if case["kind"] == "serving":
        out = serve.run(state["requests"], hbm_budget_bytes=64 << 30, max_active=48,
                        chunk_steps=case["chunk"], stream=state["stream"], keep_map=True,
                        realtime=False)["results"]
        return {"density": [out[k]["density"] for k in sorted(out)],
                "map": [out[k]["map"] for k in sorted(out)]}
    grid = state["grid"]
    if case["kind"] == "project":
        return {"map": grid.project()}
    grid.set_pulse(*state["table"])
    m, n = grid.solve_segmented() if case["kind"] == "segmented" else grid.solve()
    return {"map": m, "density": n}


# ------------------------------------------------------------------------------------------
# What a pass cannot do without, and its result in 64 bits
# ------------------------------------------------------------------------------------------

def _solve_work(c):
    pts = c["nx"] * c["ny"]
    samples = 2 if c["scheme"] == "magnus4" else 1
    return (16 * samples * c["steps"] + pts * (8 if c["precision"] == "fp64" else 4) + 8,
            pts * (FLOPS_PER_STEP * c["steps"] + FLOPS_PROJECT))


def work(case):
    if case["kind"] == "serving":
        per = [_solve_work(c) for c in _requests(case, 0)]
        return {"bytes": sum(b for b, _ in per), "flops": sum(f for _, f in per)}
    pts, elem = case["nx"] * case["ny"], 8 if case["precision"] == "fp64" else 4
    if case["kind"] == "density":
        return {"bytes": pts * elem + 8, "flops": pts}
    if case["kind"] == "project":
        return {"bytes": pts * (32 + elem), "flops": pts * FLOPS_PROJECT}
    nbytes, flops = _solve_work(case)
    return {"bytes": nbytes, "flops": flops}


def _rotate(a, b, nx, ny, nz=None):
    """psi = (a, b) <- exp(-i n.sigma) psi: n real, a component an array over the points or a
    number; a and b complex."""
    t = torch.hypot(nx, ny) if nz is None else torch.sqrt(nx * nx + ny * ny + nz * nz)
    c, s = torch.cos(t), torch.sinc(t / math.pi)  # sin(t)/t
    q = torch.complex(s * ny, s * nx)  # -i (nx - i ny) = -(ny + i nx)
    if nz is not None:
        c = torch.complex(c, -s * nz)
        return torch.addcmul(c * a, q, b, value=-1), torch.addcmul(c.conj() * b, q.conj(), a)
    return torch.addcmul(c * a, q, b, value=-1), torch.addcmul(c * b, q.conj(), a)


def _exact_solve(c):
    a, dt, a_in, a_out = _table(c)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    ex, ey, s = c["extent_x"], c["extent_y"], float(c["valley"])
    hx, hy = 2.0 * ex / c["nx"], 2.0 * ey / c["ny"]
    px = (-ex + (torch.arange(c["nx"], dtype=torch.float64, device=dev) + 0.5) * hx)[None, :]
    py = (-ey + (torch.arange(c["ny"], dtype=torch.float64, device=dev) + 0.5) * hy)[:, None]
    w = _direction(px + a_in[0], py + a_in[1], s)
    up, dn = torch.where(w == 0, torch.full_like(w, -s), -w.conj()) * math.sqrt(0.5), \
        torch.full_like(w, math.sqrt(0.5))
    wx, wy = s * dt * px, s * dt * py  # valley * dt * p
    k3, zero = math.sqrt(3.0) / 6.0, torch.zeros((), dtype=torch.float64, device=dev)
    for row in (s * dt * a).tolist():
        if c["scheme"] == "exact":
            up, dn = _rotate(up, dn, wx + row[0], wy + row[1])
        elif c["scheme"] == "strang_xy":
            half = 0.5 * (wx + row[0])
            up, dn = _rotate(up, dn, half, zero)
            up, dn = _rotate(up, dn, zero, wy + row[1])
            up, dn = _rotate(up, dn, half, zero)
        else:  # mean of the Gauss points, and their commutator along sigma_z
            x1, y1, x2, y2 = wx + row[0], wy + row[1], wx + row[2], wy + row[3]
            up, dn = _rotate(up, dn, 0.5 * (x1 + x2), 0.5 * (y1 + y2), -k3 * (x1 * y2 - y1 * x2))
    w = _direction(px + a_out[0], py + a_out[1], s)
    m = 0.5 * torch.abs(up + w.conj() * dn) ** 2
    return torch.where(w == 0, torch.zeros_like(m), m), hx * hy


def _direction(Px, Py, s):
    """valley (Px + i Py)/|P|, 0 at P = 0."""
    Px, Py = torch.broadcast_tensors(Px, Py)
    E = torch.hypot(Px, Py)
    E = torch.where(E == 0, torch.ones_like(E), E)
    return torch.complex(s * Px / E, s * Py / E)


def _too_long(cases):
    spinor_steps = sum(c["nx"] * c["ny"] * c["steps"] * (2 if c["scheme"] == "strang_xy" else 1)
                       for c in cases)
    return spinor_steps > EXACT_MOST or sum(c["steps"] for c in cases) > 150000


def exact(case, seed):
    if case["kind"] == "density":
        m = prepare(case, seed)["map"].double()
        h = 4.0 * case["extent_x"] * case["extent_y"] / (case["nx"] * case["ny"])
        return {"density": 4.0 / TWO_PI ** 2 * h * float(m.sum())}
    cases = _requests(case, seed) if case["kind"] == "serving" else [_seeded(case, seed)]
    if _too_long(cases):
        return None
    got = [_exact_solve(c) for c in cases]
    if case["kind"] == "project":
        return {"map": got[0][0]}
    density = [4.0 / TWO_PI ** 2 * h * float(m.sum()) for m, h in got]
    if case["kind"] == "serving":
        return {"density": density, "map": [m.cpu().numpy() for m, _ in got]}
    return {"map": got[0][0], "density": density[0]}
