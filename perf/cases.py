"""The work whose speed is measured: what a program that uses this library has it do.

Every case is one pass through the public entry points of ``paper_1905_07392_gb300.ebvisc``
(``Solver``, ``Batch``) on a sphere in a channel, the set-up of this repository's configurations,
tests and benchmark (``workloads.py``): box [0, nx h] x [0, ny h] x [0, nz h], inflow (0, 0, 1) at z-,
outflow at z+, slip walls in x and y (or the velocity on every side, the paper's sphere box),
seeded noise of amplitude 1e-3 on the inflow value.  Kinds:

``step``        ``advance_graph``: steps of Algorithm 1 from a given state
``host``        ``advance_host``: the same from host buffers (the end-to-end form)
``sweep``       ``Batch.advance``: a parameter sweep of independent instances
``gradient``    ``drag_gradient``: the drag and its sensitivities (adjoint, checkpointing)
``viscous``     ``solve_viscous``: the three semi-implicit viscous solves
``projection``  ``solve_projection``: the nodal projection
``derived``     ``derived``: Algorithm 2 (convective term, cell-centred projection, viscous term)
``viscosity``   ``update_viscosity``: strain rate and apparent viscosity
``monitor``     ``drag`` and ``flow_diagnostics``: what a run records between steps

Solves run to a relative residual of 1e-11 (the adjoint 1e-13, as in the benchmark): stopped
at the default 1e-8 a pressure has about seven figures and the rest follows the rounding of every
sum on the way, so results could only be compared to those seven.

The inputs come from the seed alone and are made on the GPU with torch; a pass that works in
place on device fields first copies them into the state's own buffers.
"""
import math
import random

import numpy as np
import torch

from paper_1905_07392_gb300 import ebvisc as E
from paper_1905_07392_gb300 import workloads as W

TOL = 1e-11
TOL_ADJOINT = 1e-13
CHANNEL, BOX = "channel", "box"
MODELS = {"newtonian": E.NEWTONIAN, "bingham": E.BINGHAM, "herschel_bulkley": E.HERSCHEL_BULKLEY,
          "power_law": E.POWER_LAW}
PRECISIONS = {"fp64": E.FP64, "fp32_refine": E.FP32_REFINE}


def _case(kind, nx, ny, nz, **kw):
    c = {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "radius": 0.125, "bi": 1.0, "m": 1e3, "model": "bingham",
         "n_flow": 1.0, "precision": "fp32_refine", "sides": CHANNEL, "advect": True, "steps": 1}
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: the viscosity update alone, on the 32^3 configuration, where a call is latency
        _case("viscosity", 32, 32, 32, name="viscosity_32"),
        # the same kernel on the benchmark's grid, power-law exponent in use
        _case("viscosity", 256, 256, 256, name="viscosity_256_hb", radius=0.1, m=1e4, model="herschel_bulkley",
              n_flow=0.5),
        # what a run records between steps, in the paper's sphere box [0,4D]^2 x [0,6D] at 16 cells per D
        _case("monitor", 64, 64, 96, name="monitor_box_64x64x96", bi=10.0, sides=BOX),
        # the 32^3 configuration: plain FP64, small enough that launches count
        _case("step", 32, 32, 32, name="step_32_fp64", precision="fp64", bi=0.25, steps=2),
        # the benchmark's problem on a 64^3 grid
        _case("step", 64, 64, 64, name="step_64", radius=0.1, bi=10.0, m=1e4, steps=2),
        # a ragged channel, creeping flow (the paper evaluates at Re = 1e-3, no convective term)
        _case("step", 80, 48, 112, name="step_80x48x112_creeping", bi=10.0, advect=False, steps=2),
        # the 128^3 configuration, Herschel-Bulkley n = 0.5, FP64
        _case("step", 128, 128, 128, name="step_128_fp64_hb", precision="fp64", bi=0.25, model="herschel_bulkley",
              n_flow=0.5),
        # the benchmark: 256^3, Bi = 10, m = 1e4; the second step starts from a developed pressure
        _case("step", 256, 256, 256, name="step_256", radius=0.1, bi=10.0, m=1e4, steps=2),
        # the end-to-end form: state from and to host memory every call
        _case("host", 128, 128, 128, name="host_128", bi=10.0),
        # the batched sweep of uneven grids and Bingham numbers (48^3, 64^3, 96^3)
        _case("sweep", 96, 96, 96, name="sweep_12", count=12, sweep_seed=0, radius=0.2, bi=100.0),
        # the viscous solves through their own entry point, on a large box with three different sides
        _case("viscous", 192, 160, 224, name="viscous_192x160x224", bi=10.0, m=1e4),
        # drag sensitivities: full step, two segments of checkpoints
        _case("gradient", 64, 64, 64, name="gradient_64", bi=5.0, steps=4, every=2),
    ]


def _grid(rng, lo, hi):
    """Sides that halve together down to a small bottom level: b 2^k with 3 <= b <= 7 each, the x side's size
    spread over [lo, hi] on its logarithm, the others within a factor of about two of it."""
    while True:
        want = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        k = rng.choice([k for k in range(2, 7) if 3 * 2 ** k <= 1.2 * want <= 9 * 2 ** k] or [3])
        b = [min(7, max(3, round(want * rng.uniform(0.75, 1.35) / 2 ** k))) for _ in range(3)]
        n = [v * 2 ** k for v in b]
        if (b[0] + 1) * (b[1] + 1) * (b[2] + 1) <= 512 and n[0] * n[1] * n[2] <= hi ** 3:
            return n


#: kind: how often it is drawn, and the range of its grid (cells along x; at most the upper one's cube in all)
RANGES = {"step": (6, 32, 224), "host": (1, 32, 160), "sweep": (1, 96, 96), "gradient": (1, 32, 72),
          "viscous": (2, 32, 224), "projection": (2, 32, 224), "derived": (2, 32, 256), "viscosity": (2, 32, 256),
          "monitor": (1, 32, 256)}


def draw(rng):
    kind = rng.choices(list(RANGES), [v[0] for v in RANGES.values()])[0]
    _, lo, hi = RANGES[kind]
    precision = rng.choice(["fp64", "fp32_refine", "fp32_refine"])
    if precision == "fp64" and kind in ("step", "host", "viscous", "projection", "derived"):
        hi = min(hi, 128)
    nx, ny, nz = _grid(rng, lo, hi)
    model = rng.choice(["newtonian", "bingham", "bingham", "bingham", "herschel_bulkley", "power_law"])
    if kind == "sweep":
        return _case(kind, 96, 96, 96, radius=0.2, bi=100.0, count=rng.randint(4, 14), sweep_seed=rng.randrange(1000))
    c = _case(kind, nx, ny, nz, precision=precision, model=model, m=rng.choice([1e3, 1e3, 1e4]),
              bi=0.0 if model in ("newtonian", "power_law") else round(10.0 ** rng.uniform(-1.0, 1.5), 3),
              n_flow=rng.choice([0.5, 0.75]) if model in ("herschel_bulkley", "power_law") else 1.0,
              radius=round(rng.uniform(0.1, 0.25) * min(1.0, ny / nx, nz / nx), 3), advect=rng.random() < 0.8)
    if kind in ("viscosity", "monitor", "viscous") and rng.random() < 0.3:
        c["sides"] = BOX
    if kind in ("step", "host"):
        c["steps"] = rng.choice([1, 2])
    if kind == "gradient":
        c["steps"], c["every"] = rng.choice([2, 3, 4]), 2
    return c


def _sphere(c):
    h = 1.0 / c["nx"]
    return [0.5 * c[k] * h for k in ("nx", "ny", "nz")], c["radius"], h


def _tau0(c):
    return c["bi"] / (2.0 * c["radius"])   # Bi = tau0 2r / (mu U), mu = U = 1


def _solver(c):
    centre, r, h = _sphere(c)
    s = E.Solver((c["nx"], c["ny"], c["nz"]), h, bc=W.CHANNEL_BC if c["sides"] == CHANNEL else (W.INFLOW,) * 6,
                 u_in=(0.0, 0.0, 1.0), tau0=_tau0(c), m=c["m"], n_flow=c["n_flow"], model=MODELS[c["model"]],
                 bi_cfl=c["bi"], tol=TOL_ADJOINT if c["kind"] == "gradient" else TOL, max_iters=5000,
                 precision=PRECISIONS[c["precision"]], advect=int(c["advect"]))
    s.build_spheres([centre + [r]])
    return s


def _coords(c, nodes=False):
    """x, y, z of the cell centres (or nodes), shaped to broadcast as (z, y, x)."""
    h, off = 1.0 / c["nx"], 0.0 if nodes else 0.5
    ax = [(torch.arange(c[k] + int(nodes), dtype=torch.float64, device="cuda") + off) * h for k in ("nx", "ny", "nz")]
    return ax[0][None, None, :], ax[1][None, :, None], ax[2][:, None, None]


def _fluid(c):
    """1.0 in cells that hold fluid (some corner outside the sphere), 0.0 in covered ones: a cell lies inside the
    (convex) sphere if and only if all its corners do."""
    centre, r, _ = _sphere(c)
    x, y, z = _coords(c, nodes=True)
    out = torch.sqrt((x - centre[0]) ** 2 + (y - centre[1]) ** 2 + (z - centre[2]) ** 2) - r > 0
    f = torch.zeros((c["nz"], c["ny"], c["nx"]), dtype=torch.bool, device="cuda")
    for q in range(8):
        i, j, k = q & 1, (q >> 1) & 1, q >> 2
        f |= out[k:k + c["nz"], j:j + c["ny"], i:i + c["nx"]]
    return f.to(torch.float64)


def _noise(shape, seed, salt=0):
    g = torch.Generator(device="cuda")
    g.manual_seed(1009 * int(seed) + salt)
    return torch.rand(shape, generator=g, device="cuda", dtype=torch.float64) * 2.0 - 1.0


def _velocity(c, seed, disturbed):
    """(3, nz, ny, nx): the inflow value plus noise of 1e-3; disturbed: also the dipole of a sphere moving through it
    and a smooth disturbance of random phase, a state as a run has it after some steps."""
    u = 1e-3 * _noise((3, c["nz"], c["ny"], c["nx"]), seed)
    u[2] += 1.0
    if disturbed:
        centre, r, _ = _sphere(c)
        x, y, z = _coords(c)
        X, Y, Z = x - centre[0], y - centre[1], z - centre[2]
        d2 = (X * X + Y * Y + Z * Z).clamp_min((0.5 * r) ** 2)
        a = 0.5 * r ** 3 * d2 ** -2.5
        u[0] -= 3.0 * a * X * Z
        u[1] -= 3.0 * a * Y * Z
        u[2] += a * (d2 - 3.0 * Z * Z)
        ph = random.Random(seed).uniform(0.0, 6.28)
        u[0] += 0.05 * torch.sin(2 * math.pi * x) * torch.cos(2 * math.pi * (y + z) + ph)
        u[1] += 0.05 * torch.sin(2 * math.pi * y) * torch.cos(2 * math.pi * (z - x) + ph)
        u[2] += 0.05 * torch.cos(2 * math.pi * (x - y) + ph)
    return u * _fluid(c)


def _pressure(c, seed):
    x, y, z = _coords(c, nodes=True)
    ph = random.Random(seed + 7).uniform(0.0, 6.28)
    L = c["nz"] / c["nx"]
    return ((L - z) * (1.0 + 0.2 * torch.sin(2 * math.pi * (x + y) + ph))).contiguous()


def _eta(c, seed):
    """Viscosity of a flow that yields near the body and is nearly rigid far from it."""
    centre, r, _ = _sphere(c)
    x, y, z = _coords(c)
    d = torch.sqrt((x - centre[0]) ** 2 + (y - centre[1]) ** 2 + (z - centre[2]) ** 2).clamp_min(0.5 * r)
    ph = random.Random(seed + 13).uniform(0.0, 6.28)
    s = (r / d) ** 4 / r * (1.0 + 0.3 * torch.sin(6.28 * (x + 2 * y - z) + ph))
    if c["model"] == "newtonian":
        eta = torch.ones_like(s)
    else:
        visc = s.clamp_min(1.0 / c["m"]) ** (c["n_flow"] - 1.0)
        eta = visc + _tau0(c) * -torch.expm1(-c["m"] * s) / s
    return eta * _fluid(c)


def _dt(c):
    h = 1.0 / c["nx"]
    return 0.5 * h * h / (6.0 * (1.0 + c["bi"]))   # the viscous limit of the library's own time step


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "sweep":
        ws = W.batched_sweep(c["sweep_seed"], c["count"])
        b = E.Batch(ws, precision=E.FP32_REFINE, tol=TOL, max_iters=5000)
        b.build_spheres()
        u0, p0 = [], []
        for q, w in enumerate(ws):
            u = 1e-3 * _noise((3, w.n ** 3), seed, q)
            u[2] += 1.0
            u0.append((u * (b.instance(q).geometry()["alpha"] > 0)).reshape(-1).contiguous())
            p0.append(torch.zeros(b.instance(q).nnode, dtype=torch.float64, device="cuda"))
        return {"case": c, "batch": b, "u0": u0, "p0": p0, "u": [t.clone() for t in u0],
                "p": [t.clone() for t in p0]}
    s = _solver(c)
    st = {"case": c, "solver": s}
    new = lambda n: torch.empty(n, dtype=torch.float64, device="cuda")  # noqa: E731
    if kind in ("step", "host", "gradient"):
        st["u0"] = _velocity(c, seed, False).reshape(-1).contiguous()
        st["p0"] = torch.zeros(s.nnode, dtype=torch.float64, device="cuda")
        st["u"], st["p"] = st["u0"].clone(), st["p0"].clone()
        if kind == "host":   # (its passes go on from each other, as a run's steps do)
            st["u"], st["p"] = st["u"].cpu().pin_memory(), st["p"].cpu().pin_memory()
        if kind == "gradient":
            st["f"] = 0.1 * _noise(3 * s.ncell, seed, 5)
        return st
    if kind == "viscous":
        st["eta"] = _eta(c, seed).reshape(-1).contiguous()
        st["psi"] = _velocity(c, seed, True).reshape(-1).contiguous()
        st["ut"] = new(3 * s.ncell)
    elif kind == "projection":
        st["u0"] = _velocity(c, seed, True).reshape(-1).contiguous()
        st["p0"] = _pressure(c, seed).reshape(-1).contiguous()
        st["u"], st["p"] = st["u0"].clone(), st["p0"].clone()
    else:
        st["u"] = _velocity(c, seed, True).reshape(-1).contiguous()
        if kind == "derived":
            st["C"], st["eta"], st["V"] = new(3 * s.ncell), new(s.ncell), new(3 * s.ncell)
        elif kind == "viscosity":
            st["eta"], st["srate"] = new(s.ncell), new(s.ncell)
        else:
            st["p"] = _pressure(c, seed).reshape(-1).contiguous()
            st["lam"], st["dev"] = new(s.ncell), new(s.ncell)
    return st


def run(state):
    c, kind = state["case"], state["case"]["kind"]
    if kind == "sweep":
        for a in ("u", "p"):
            for t, t0 in zip(state[a], state[a + "0"]):
                t.copy_(t0)
        st = state["batch"].advance(state["u"], state["p"], steps=1)
        return {"u": state["u"], "p": state["p"], "drag": [x["drag"] for x in st]}
    s = state["solver"]
    if kind in ("step", "projection"):
        state["u"].copy_(state["u0"])
        state["p"].copy_(state["p0"])
    if kind == "step":
        st = s.advance_graph(state["u"], state["p"], steps=c["steps"])
        return {"u": state["u"], "p": state["p"], "dt": st["dt"], "drag": st["drag"], "yielded": st["yield_frac"]}
    if kind == "host":
        st = s.advance_host(state["u"].numpy(), state["p"].numpy(), steps=c["steps"])
        return {"u": state["u"], "p": state["p"], "dt": st["dt"], "drag": st["drag"], "yielded": st["yield_frac"]}
    if kind == "gradient":
        J, gt, gm, fb = s.drag_gradient(state["u0"], state["p0"], _dt(c), c["steps"], c["every"], f=state["f"])
        return {"J": J, "dtau0": gt, "dmu": gm, "df": fb}
    if kind == "viscous":
        s.solve_viscous(state["eta"], state["psi"], _dt(c), state["ut"])
        return {"ut": state["ut"]}
    if kind == "projection":
        s.solve_projection(state["u"], state["p"], _dt(c))
        return {"u": state["u"], "p": state["p"]}
    if kind == "derived":
        s.derived(state["u"], state["C"], state["eta"], state["V"])
        return {"C": state["C"], "eta": state["eta"], "V": state["V"]}
    if kind == "viscosity":
        s.update_viscosity(state["u"], state["eta"], state["srate"])
        return {"eta": state["eta"], "srate": state["srate"]}
    fz, yf = s.drag(state["u"], state["p"])
    s.flow_diagnostics(state["u"], state["lam"], state["dev"])
    return {"drag": fz, "yielded": yf, "lam": state["lam"], "dev": state["dev"]}


# words read and written per cell, and operations per cell that the path cannot do without: one
# application of each operator and one evaluation of each explicit term (no solver iterations)
_WORDS = {"step": (4, 4), "host": (4, 4), "gradient": (7, 3), "viscous": (4, 3), "projection": (4, 4),
          "derived": (3, 7), "viscosity": (3, 2), "monitor": (4, 2)}
_FLOPS = {"step": 800, "host": 800, "gradient": 2400, "viscous": 60, "projection": 100, "derived": 250,
          "viscosity": 40, "monitor": 60}


def work(case):
    c = case
    if c["kind"] == "sweep":
        cells = sum(w.n ** 3 for w in W.batched_sweep(c["sweep_seed"], c["count"]))
        return {"bytes": 8.0 * 8 * cells, "flops": 800.0 * cells}
    cells = c["nx"] * c["ny"] * c["nz"]
    times = c["steps"] if c["kind"] in ("step", "host", "gradient") else 1
    return {"bytes": 8.0 * sum(_WORDS[c["kind"]]) * cells, "flops": float(_FLOPS[c["kind"]]) * cells * times}


def _gradients(c, u):
    """G[d][q] = d u_q / d x_d on the cells: central where both neighbours hold fluid, one-sided quadratic next to a
    covered cell or the box side, first order with one neighbour, zero with none."""
    ok = _fluid(c) > 0
    ih = float(c["nx"])

    def shift(a, d, k):
        # the value k cells along axis d (x: last), False / 0 outside the box
        ax = 2 - d
        out = torch.zeros_like(a)
        n = a.shape[ax]
        if abs(k) < n:
            out.narrow(ax, max(0, -k), n - abs(k)).copy_(a.narrow(ax, max(0, k), n - abs(k)))
        return out

    G = [[None] * 3 for _ in range(3)]
    for d in range(3):
        p1, m1 = shift(ok, d, 1), shift(ok, d, -1)
        p2, m2 = shift(ok, d, 2), shift(ok, d, -2)
        for q in range(3):
            f = u[q]
            fp, fm, fpp, fmm = (shift(f, d, k) for k in (1, -1, 2, -2))
            g = torch.zeros_like(f)
            g = torch.where(p1 & ~m1, torch.where(p2, -1.5 * f + 2.0 * fp - 0.5 * fpp, fp - f), g)
            g = torch.where(m1 & ~p1, torch.where(m2, 0.5 * fmm - 2.0 * fm + 1.5 * f, f - fm), g)
            g = torch.where(p1 & m1, 0.5 * (fp - fm), g)
            G[d][q] = g * ih
    return G, ok


def _strain(c, G, ok):
    s = 2.0 * (G[0][0] ** 2 + G[1][1] ** 2 + G[2][2] ** 2)
    for a, b in ((0, 1), (0, 2), (1, 2)):
        s = s + (G[a][b] + G[b][a]) ** 2
    sr = torch.sqrt(s)
    tau0, floor = _tau0(c), sr.clamp_min(1.0 / c["m"])
    plastic = tau0 * torch.where(sr > 0, -torch.expm1(-c["m"] * sr) / sr, torch.full_like(sr, c["m"]))
    power = floor ** (c["n_flow"] - 1.0)
    eta = {"newtonian": torch.ones_like(sr), "bingham": 1.0 + plastic, "herschel_bulkley": power + plastic,
           "power_law": power}[c["model"]]
    return sr * ok, eta * ok, s


def exact(case, seed):
    c = case
    if c["kind"] not in ("viscosity", "monitor"):
        return None   # a linear solve on the cut-cell operators: not a formula to write down a second time
    u = _velocity(c, seed, True)
    G, ok = _gradients(c, u)
    sr, eta, s = _strain(c, G, ok)
    if c["kind"] == "viscosity":
        return {"eta": eta.reshape(-1), "srate": sr.reshape(-1)}
    w2 = (G[1][2] - G[2][1]) ** 2 + (G[2][0] - G[0][2]) ** 2 + (G[0][1] - G[1][0]) ** 2
    lam = torch.where(s + w2 > 0, (s - w2) / (s + w2), torch.zeros_like(s)) * ok
    tau0 = _tau0(c)
    dev = (eta * sr / tau0 - 1.0) * ok if tau0 > 0 else torch.zeros_like(s)
    return {"drag": None, "yielded": None, "lam": lam.reshape(-1), "dev": dev.reshape(-1)}
