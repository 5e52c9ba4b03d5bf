"""Performance cases of the extended lattice Boltzmann library.

A case is one call sequence that a program using the library makes, on inputs
that are already on the GPU:

  solve     initialise from density and velocity, advance a number of steps,
            read density and velocity back (the loop of every run);
  restart   load populations, advance, read the populations back (checkpoint
            and restart, coupling to another code);
  served    one chunk of the served mix: the resident solves grouped by storage
            and kernel form, one batched call for each group, then every
            solve's density and velocity;
  diagnose  the FP64 reductions and the Fourier-mode amplitude of a running
            solve, as a program takes them every few steps.

``listed`` gives the cases, ``draw`` more of the same ranges, ``prepare`` and
``run`` one pass, ``work`` the bytes and operations a pass cannot do without,
and ``exact`` the same results in FP64 with torch operations only.
"""
from __future__ import annotations

import math

import torch

from paper_2101_04550_gb300 import elbm

THIRD = 1.0 / 3.0
ELEMENT_BYTES = {"f32": 4, "f32s": 4, "f16": 2, "bf16": 2}
# node updates of one drawn pass at most: below the largest listed cases
DRAW_UPDATES = {2: 2.0e8, 3: 1.0e8}


# ------------------------------------------------------------------- cases
def _case(name, kind, n, steps, storage, field, lam=(1.0, 1.0, 1.0), T=THIRD, omega=1.8, speed=0.0,
          walls=False, force=0.0, kernel=0, equilibrium=0):
    """One case as plain values.  Grids are given as nx, ny, nz with nz = 1 for
    D2Q9; ``speed`` is a uniform advection added to the field and taken as the
    storage baseline velocity, as the served mix does."""
    c = {"kind": kind, "nx": n[0], "ny": n[1], "nz": n[2], "steps": steps, "storage": storage, "field": field,
         "lam_x": lam[0], "lam_y": lam[1], "lam_z": lam[2], "T": T, "omega": omega, "speed": speed,
         "walls": walls, "force": force, "kernel": kernel, "equilibrium": equilibrium}
    if name:
        c = {"name": name, **c}
    return c


def listed():
    return [
        # the advected shear wave on which the viscosity is measured: a tiny
        # grid and many steps, so launches and latency are all there is
        _case("shear2d_64", "solve", (64, 64, 1), 200, "f32", "shear", omega=2.0 / 1.06, speed=0.1),
        # the stretched double shear layer of the validation runs (L2-resident)
        _case("dsl2d_1024x512", "solve", (1024, 512, 1), 100, "f32", "dsl", lam=(1.0, 2.0, 1.0), T=0.5, omega=1.9),
        # the same flow well beyond the L2 cache
        _case("dsl2d_4096", "solve", (4096, 4096, 1), 20, "f32", "dsl", T=0.5, omega=1.9),
        # the smallest solve of the served mix, alone
        _case("shear3d_32", "solve", (32, 32, 32), 100, "f32s", "shear", T=0.45, speed=0.1),
        # a middle-sized solve of the served mix, alone, in half-precision storage
        _case("tg3d_96_f16", "solve", (96, 96, 96), 50, "f16", "taylor_green", T=0.4, speed=0.15),
        # decaying turbulence on 256^3, the benchmark flow, in its two storages
        _case("turbulence_256", "solve", (256, 256, 256), 20, "f32s", "modes"),
        _case("turbulence_256_f16", "solve", (256, 256, 256), 20, "f16", "modes"),
        # the wall-bounded channel with its body force on the stretched lattice
        _case("channel_512x128x256", "solve", (512, 128, 256), 10, "f32", "channel", lam=(2.0, 1.0, 2.0), T=0.55,
              walls=True, force=4e-7),
        # a box whose sizes suit no tile, one population array, stepped between
        # checkpoints
        _case("restart_135x121x150", "restart", (135, 121, 150), 20, "f32", "modes", lam=(1.0, 1.5, 2.0), T=0.45),
        # the two-array form asked for on a box that is no multiple of the tiles
        _case("box_180x120x100", "solve", (180, 120, 100), 20, "f32s", "modes", T=0.4, kernel=3),
        # one scheduling chunk of the served mix: every size, both storages
        _case("served_chunk", "served", (128, 128, 128), 50, "mixed", "mixed", T=0.4, speed=0.1),
        # the FP64 reductions (energy, enstrophy, extrema) and the mode
        # amplitude of a turbulence run
        _case("diagnose_256", "diagnose", (256, 256, 256), 4, "f32s", "modes", speed=0.05),
    ]


# the resident solves of the served chunk: sizes of the mix with their stretch
MIX = [((32, 32, 32), 1.0), ((48, 48, 48), 1.0), ((64, 64, 64), 1.0), ((64, 32, 64), 2.0),
       ((96, 96, 96), 1.0), ((128, 128, 128), 1.0)]


def members(case):
    """The solves of a served chunk: every size up to the case's largest, in
    FP32 and in FP16 shifted storage."""
    out = []
    for k, (n, lam_y) in enumerate(MIX):
        if n[0] > case["nx"]:
            continue
        for storage in ("f32s", "f16"):
            # single pass where the grid allows it, two-pass otherwise, as the server chooses
            kernel = 3 if n[0] % 32 == 0 and n[1] % 16 == 0 else 1
            out.append(_case(None, "solve", n, case["steps"], storage, ("shear", "taylor_green")[k % 2],
                             lam=(1.0, lam_y, 1.0), T=case["T"], omega=case["omega"] - 0.02 * k,
                             speed=case["speed"], kernel=kernel))
    return out


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_steps(rng, nodes, dims, hi):
    most = max(2, min(hi, int(DRAW_UPDATES[dims] / nodes)))
    return rng.randint(max(2, most // 2), most)


def draw(rng):
    kind = rng.choice(["flow2d", "flow2d", "flow3d", "flow3d", "flow3d", "channel", "restart", "single", "served",
                       "diagnose"])
    T = rng.uniform(0.3, 0.55)
    omega = rng.uniform(1.5, 1.9)
    storage = rng.choice(["f32", "f32s", "f16", "bf16"])
    if kind == "flow2d":
        nx, ny = _log_uniform(rng, 33, 4000), _log_uniform(rng, 33, 4000)
        lam = (1.0, rng.choice([1.0, 1.5, 2.0]), 1.0)
        return _case(None, "solve", (nx, ny, 1), _draw_steps(rng, nx * ny, 2, 200), storage,
                     rng.choice(["shear", "dsl", "modes"]), lam=lam, T=T, omega=omega,
                     equilibrium=rng.choice([0, 0, 0, 1]))
    if kind == "served":
        return _case(None, "served", (rng.choice([48, 64, 96]),) * 3, rng.randint(20, 60), "mixed", "mixed", T=T,
                     omega=rng.uniform(1.6, 1.85), speed=rng.uniform(0.02, 0.12))
    if kind == "flow3d":
        # the sizes programs choose: multiples of 16 or 32
        n = tuple(s * max(1, _log_uniform(rng, 24, 230) // s) for s in (32, 16, 1))
    else:
        n = tuple(_log_uniform(rng, 20, 200) for _ in range(3))
    lam = tuple(rng.choice([1.0, 1.0, 1.5, 2.0]) for _ in range(3))
    nodes = n[0] * n[1] * n[2]
    if kind == "channel":
        n = (32 * max(1, n[0] // 32), 16 * max(1, n[1] // 16), n[2])
        nodes = n[0] * n[1] * n[2]
        return _case(None, "solve", n, _draw_steps(rng, nodes, 3, 100), storage, "channel", lam=(2.0, 1.0, 2.0), T=T,
                     omega=omega, walls=True, force=rng.uniform(1e-7, 1e-6))
    if kind == "diagnose":
        return _case(None, "diagnose", n, rng.randint(1, 4), storage, "modes", lam=lam, T=T, omega=omega,
                     speed=rng.uniform(0.02, 0.08), walls=rng.choice([False, True]))
    return _case(None, "restart" if kind == "restart" else "solve", n, _draw_steps(rng, nodes, 3, 100), storage,
                 rng.choice(["shear", "taylor_green", "modes"]), lam=lam, T=T, omega=omega,
                 speed=rng.choice([0.0, rng.uniform(0.02, 0.1)]), kernel=3 if kind == "single" else 0,
                 equilibrium=rng.choice([0, 0, 0, 1, 2]) if kind == "restart" and storage.startswith("f32") else 0)


# ------------------------------------------------------------------ inputs
def _grid(case):
    """(D, field shape, lam, physical coordinates x, y, z broadcastable to the shape)."""
    n = (case["nx"], case["ny"], case["nz"])
    lam = (case["lam_x"], case["lam_y"], case["lam_z"])
    D = 2 if case["nz"] == 1 else 3
    shape = tuple(n[:D][::-1])
    X = []
    for a in range(D):
        v = torch.arange(n[a], dtype=torch.float64, device="cuda") * lam[a]
        X.append(v.reshape([-1 if d == D - 1 - a else 1 for d in range(D)]))
    return D, shape, lam, X


def _advection(case, D):
    return [v * case["speed"] for v in (0.64, 0.6, 0.48)][:D]


def _field(case, seed):
    """rho and u (float32, on the GPU) of the case's flow."""
    D, shape, lam, X = _grid(case)
    n = (case["nx"], case["ny"], case["nz"])
    g = torch.Generator().manual_seed(seed)

    def rand():
        return float(torch.rand((), generator=g, dtype=torch.float64))

    k1 = [2.0 * math.pi / (n[a] * lam[a]) for a in range(D)]
    u = torch.zeros((D,) + shape, dtype=torch.float64, device="cuda")
    kind = case["field"]
    if kind == "shear":  # a plane wave along a lattice diagonal, transverse velocity
        phase = k1[0] * X[0] + k1[1] * X[1] + 2.0 * math.pi * rand()
        norm = math.hypot(k1[0], k1[1])
        amp = 1e-2 * (0.5 + rand())
        u[0] += -k1[1] / norm * amp * torch.sin(phase)
        u[1] += k1[0] / norm * amp * torch.sin(phase)
    elif kind == "taylor_green":
        px, py = 2.0 * math.pi * rand(), 2.0 * math.pi * rand()
        amp = 0.02 * (0.5 + rand())
        env = torch.cos(k1[2] * X[2]) if D == 3 else 1.0
        u[0] += amp * torch.sin(k1[0] * X[0] + px) * torch.cos(k1[1] * X[1] + py) * env
        u[1] += -amp * k1[0] / k1[1] * torch.cos(k1[0] * X[0] + px) * torch.sin(k1[1] * X[1] + py) * env
    elif kind == "dsl":  # two shear layers in y, a small wave in x
        yn, xn = X[1] / (n[1] * lam[1]), X[0] / (n[0] * lam[0])
        u[0] += torch.where(yn <= 0.5, torch.tanh(80.0 * (yn - 0.25)), torch.tanh(80.0 * (0.75 - yn))) * 0.1
        u[1] += 0.005 * torch.sin(2.0 * math.pi * (xn + rand()))
    elif kind == "channel":  # laminar profile and a random perturbation of 5 %
        yc = (torch.arange(n[1], dtype=torch.float64, device="cuda") + 0.5) / n[1]
        u[0] += (0.4 * yc * (1.0 - yc)).reshape(1, -1, 1)
        gd = torch.Generator(device="cuda").manual_seed(seed)
        u += 0.005 * (2.0 * torch.rand(u.shape, generator=gd, dtype=torch.float64, device="cuda") - 1.0)
    else:  # random solenoidal modes of the largest scales (one of them the box
        # diagonal, whose amplitude the diagnostics follow), u_rms 0.05 per component
        for j in range(8):
            m = [1 + int(4 * rand()) if a == 0 else int(9 * rand()) - 4 for a in range(D)]
            if j == 0:
                m = [1, 1, 0][:D]
            k = [m[a] * k1[a] for a in range(D)]
            s = [rand() + 0.1 if a == 0 else -rand() - 0.1 if a == 1 else rand() - 0.5 for a in range(D)]
            kk = sum(v * v for v in k)
            dot = sum(k[a] * s[a] for a in range(D)) / kk
            s = [s[a] - dot * k[a] for a in range(D)]
            norm = math.sqrt(sum(v * v for v in s)) + 1e-9
            wave = torch.sin(sum(k[a] * X[a] for a in range(D)) + 2.0 * math.pi * rand())
            for a in range(D):
                u[a] += 0.043 * s[a] / norm * wave
    for a, v in enumerate(_advection(case, D)):
        u[a] += v
    rho = torch.ones(shape, dtype=torch.float64, device="cuda")
    return rho.float(), u.float()


def _nu(case):
    return (1.0 / case["omega"] - 0.5) * case["T"]


def _solver(case):
    D = 2 if case["nz"] == 1 else 3
    shifted = case["storage"] != "f32" and case["speed"] != 0.0
    return elbm.Solver(elbm.D2Q9 if D == 2 else elbm.D3Q27, (case["nx"], case["ny"], case["nz"])[:D],
                       stretch=(case["lam_x"], case["lam_y"], case["lam_z"]), T=case["T"], nu=_nu(case),
                       storage=case["storage"], stream=torch.cuda.current_stream(), kernel=case["kernel"],
                       equilibrium=case["equilibrium"], walls_y=case["walls"],
                       u_ref=_advection(case, D) if shifted and case["equilibrium"] != 2 else None,
                       force=(case["force"], 0.0, 0.0)[:D] if case["force"] else None)


def _wavevector(case):
    return (2.0 * math.pi / (case["nx"] * case["lam_x"]), 2.0 * math.pi / (case["ny"] * case["lam_y"]), 0.0)


def prepare(case, seed):
    if case["kind"] == "served":
        ms = members(case)
        state = {"kind": "served", "steps": case["steps"], "solvers": [], "fields": [], "outs": [], "batches": []}
        groups = {}
        for k, m in enumerate(ms):
            s = _solver(m)
            rho, u = _field(m, seed + 1000 * k)
            s.init(rho, u)
            state["solvers"].append(s)
            state["fields"].append((rho, u))
            state["outs"].append((torch.empty_like(rho), torch.empty_like(u)))
            groups.setdefault((m["storage"], m["kernel"]), []).append(s)
        state["batches"] = [elbm.Batch(g) for g in groups.values()]
        return state
    s = _solver(case)
    rho, u = _field(case, seed)
    state = {"kind": case["kind"], "steps": case["steps"], "solver": s}
    if case["kind"] == "solve":
        state.update(rho=rho, u=u, rho_out=torch.empty_like(rho), u_out=torch.empty_like(u))
    elif case["kind"] == "restart":
        f = _equilibrium(case, rho.double(), u.double()).float()
        state.update(f=f, f_out=torch.empty_like(f))
    else:
        s.init(rho, u)
        s.step(case["steps"])
        state.update(k=_wavevector(case), direction=(0.0, 1.0, 0.0))
    return state


def run(state):
    if state["kind"] == "solve":
        s = state["solver"]
        s.init(state["rho"], state["u"])
        s.step(state["steps"])
        s.moments(state["rho_out"], state["u_out"])
        return state["rho_out"], state["u_out"]
    if state["kind"] == "restart":
        s = state["solver"]
        s.set_populations(state["f"])
        s.step(state["steps"])
        s.get_populations(state["f_out"])
        return state["f_out"]
    if state["kind"] == "served":
        for s, (rho, u) in zip(state["solvers"], state["fields"]):
            s.init(rho, u)
        for b in state["batches"]:
            b.step(state["steps"])
        for s, (rho, u) in zip(state["solvers"], state["outs"]):
            s.moments(rho, u)
        return [t for pair in state["outs"] for t in pair]
    sums = state["solver"].reduce()
    sums["amplitude"] = state["solver"].mode_amplitude(state["k"], state["direction"])
    return sums


# -------------------------------------------------------------------- work
def work(case):
    """Bytes and operations of one pass.  A time step reads and writes every
    population once; initialisation writes them and reads rho and u; the
    read-outs read them and write theirs.  Operations per node and step: the
    moments (3 Q additions), the product-form equilibrium (3 per population),
    its difference from the population and the relaxation (3 per population),
    and about 30 for the anomaly, its differences and the axis factors."""
    if case["kind"] == "served":
        parts = [work(m) for m in members(case)]
        return {"bytes": sum(p["bytes"] for p in parts), "flops": sum(p["flops"] for p in parts)}
    D = 2 if case["nz"] == 1 else 3
    Q = 9 if D == 2 else 27
    N = case["nx"] * case["ny"] * case["nz"]
    es = ELEMENT_BYTES[case["storage"]]
    pops, macro = Q * es * N, 4 * (1 + D) * N
    if case["kind"] == "diagnose":  # two read-outs (the reductions, the mode sums) of the populations
        return {"bytes": 2 * pops, "flops": (6 * Q + 60) * N}
    ends = 2 * (pops + (4 * Q * N if case["kind"] == "restart" else macro))
    return {"bytes": case["steps"] * 2 * pops + ends, "flops": case["steps"] * (9 * Q + 30) * N}


# ------------------------------------------------------- FP64 reference
def _directions(D):
    return [(cx, cy, cz) for cz in ((0,) if D == 2 else (-1, 0, 1)) for cy in (-1, 0, 1) for cx in (-1, 0, 1)]


def _triplet(u, P, lam):
    """Psi_c for c = -1, 0, 1 along one axis."""
    s = P / (lam * lam)
    return 0.5 * (s - u / lam), 1.0 - s, 0.5 * (s + u / lam)


def _products(case, rho, u, P):
    """Generator of (i, rho prod_a Psi_a) over the populations."""
    D = u.shape[0]
    lam = (case["lam_x"], case["lam_y"], case["lam_z"])
    tri = [_triplet(u[a], P[a], lam[a]) for a in range(D)]
    for i, c in enumerate(_directions(D)):
        f = rho * tri[0][c[0] + 1] * tri[1][c[1] + 1]
        yield i, (f * tri[2][c[2] + 1] if D == 3 else f)


def _second_order(case, rho, u):
    """The product form with every term above second order in u dropped."""
    D = u.shape[0]
    lam = (case["lam_x"], case["lam_y"], case["lam_z"])
    T = case["T"]
    for i, c in enumerate(_directions(D)):
        A, B, C = [], [], []
        for a in range(D):
            w = T / lam[a] ** 2
            A.append(1.0 - w if c[a] == 0 else 0.5 * w)
            B.append(0.5 * c[a] / lam[a])
            C.append(-1.0 / lam[a] ** 2 if c[a] == 0 else 0.5 / lam[a] ** 2)
        total = math.prod(A)
        for a in range(D):
            rest = math.prod(A[b] for b in range(D) if b != a)
            total = total + rest * (B[a] * u[a] + C[a] * u[a] ** 2)
            for b in range(a + 1, D):
                rest2 = math.prod(A[d] for d in range(D) if d not in (a, b))
                total = total + rest2 * B[a] * B[b] * u[a] * u[b]
        yield i, rho * total


def _equilibrium(case, rho, u):
    P = [case["T"] + u[a] ** 2 for a in range(u.shape[0])]
    return torch.stack([f for _, f in _products(case, rho, u, P)])


def _macros(case, f):
    D = 2 if case["nz"] == 1 else 3
    lam = (case["lam_x"], case["lam_y"], case["lam_z"])
    rho = f.sum(0)
    u = torch.zeros((D,) + rho.shape, dtype=f.dtype, device=f.device)
    for i, c in enumerate(_directions(D)):
        for a in range(D):
            if c[a]:
                u[a] += c[a] * lam[a] * f[i]
    return rho, u / rho


def _difference(case, v, a, axis_is_y_wall):
    """Central difference along axis a (node spacing lam_a); beyond a wall the
    negated value of the wall-adjacent node."""
    dim = v.dim() - 1 - a
    lam = (case["lam_x"], case["lam_y"], case["lam_z"])
    up, dn = torch.roll(v, -1, dim), torch.roll(v, 1, dim)
    if axis_is_y_wall:
        last = v.shape[dim] - 1
        up.narrow(dim, last, 1).copy_(-v.narrow(dim, last, 1))
        dn.narrow(dim, 0, 1).copy_(-v.narrow(dim, 0, 1))
    return (up - dn) / (2.0 * lam[a])


def _step(case, f):
    D = 2 if case["nz"] == 1 else 3
    lam = (case["lam_x"], case["lam_y"], case["lam_z"])
    T, om, walls = case["T"], 1.0 / (_nu(case) / case["T"] + 0.5), case["walls"]
    rho, u = _macros(case, f)
    if case["equilibrium"] == 2:
        eq = _second_order(case, rho, u)
    else:
        P = []
        for a in range(D):
            p = T + u[a] ** 2
            if case["equilibrium"] == 0:
                q = rho * u[a] * (lam[a] ** 2 - 3.0 * T - u[a] ** 2)
                p = p + (2.0 - om) / (2.0 * om) * _difference(case, q, a, walls and a == 1) / rho
            P.append(p)
        eq = _products(case, rho, u, P)
    forced = [None] * (9 if D == 2 else 27)
    if case["force"]:
        ug = u.clone()
        ug[0] += case["force"]
        plain = _products(case, rho, u, [T + u[a] ** 2 for a in range(D)])
        moved = _products(case, rho, ug, [T + ug[a] ** 2 for a in range(D)])
        forced = (b - a for (_, a), (_, b) in zip(plain, moved))
    out = torch.empty_like(f)
    Q = f.shape[0]
    dirs = _directions(D)
    for (i, feq), extra in zip(eq, forced):
        post = f[i] + om * (feq - f[i])
        if extra is not None:
            post = post + extra
        c = dirs[i]
        for a in range(D):
            if c[a] and not (walls and a == 1):
                post = torch.roll(post, c[a], post.dim() - 1 - a)
        if walls and c[1]:
            # moved along x and z above; along y without wrapping, and what
            # would cross a wall returns reversed to the node it left
            dim = post.dim() - 2
            ny = post.shape[dim]
            src, dst = (0, 1) if c[1] > 0 else (1, 0)
            out[i].narrow(dim, dst, ny - 1).copy_(post.narrow(dim, src, ny - 1))
            edge = ny - 1 if c[1] > 0 else 0
            stay = f[i].narrow(dim, edge, 1) + om * (feq.narrow(dim, edge, 1) - f[i].narrow(dim, edge, 1))
            if extra is not None:
                stay = stay + extra.narrow(dim, edge, 1)
            out[Q - 1 - i].narrow(dim, edge, 1).copy_(stay)
        else:
            out[i] = post
    return out


def _exact_sums(case, f):
    """The reductions of a state, named as the library names them."""
    D = 2 if case["nz"] == 1 else 3
    walls = case["walls"]
    rho, u = _macros(case, f)
    w = torch.zeros((3,) + rho.shape, dtype=f.dtype, device=f.device)
    w[:D] = u
    w[0] += 0.5 * case["force"]

    def dif(v, a):
        return _difference(case, v, a, walls and a == 1) if a < D else torch.zeros_like(v)

    curl2 = (dif(w[1], 0) - dif(w[0], 1)) ** 2
    if D == 3:
        curl2 = curl2 + (dif(w[2], 1) - dif(w[1], 2)) ** 2 + (dif(w[0], 2) - dif(w[2], 0)) ** 2
    u2 = (w ** 2).sum(0)
    wall = 0.0
    if walls:
        dim = rho.dim() - 2
        ny = rho.shape[dim]
        for first, second in ((0, 1), (ny - 1, ny - 2)):
            wall += float((9.0 * w[0].select(dim, first) - w[0].select(dim, second)).sum()) / (3.0 * case["lam_y"])
    k = _wavevector(case)
    _, _, _, X = _grid(case)
    phase = k[0] * X[0] + k[1] * X[1]
    amp = math.hypot(float((w[1] * torch.cos(phase)).sum()), float((w[1] * torch.sin(phase)).sum()))
    return {"mass": float(rho.sum()), "mom_x": float((rho * w[0]).sum()), "mom_y": float((rho * w[1]).sum()),
            "mom_z": float((rho * w[2]).sum()), "rho_u2": float((rho * u2).sum()), "u2": float(u2.sum()),
            "curl2": float(curl2.sum()), "dxux2": float((dif(w[0], 0) ** 2).sum()),
            "ux2": float((w[0] ** 2).sum()), "fmin": float(f.min()), "nonfinite": 0.0,
            "umax": float(u2.sqrt().max()), "wall_dudn": wall, "amplitude": 2.0 * amp / rho.numel()}


def exact(case, seed):
    if case["kind"] == "served":
        out = []
        for k, m in enumerate(members(case)):
            out.extend(exact(m, seed + 1000 * k))
        return out
    rho, u = _field(case, seed)
    f = _equilibrium(case, rho.double(), u.double())
    if case["kind"] == "restart":
        f = f.float().double()
    for _ in range(case["steps"]):
        f = _step(case, f)
    if case["kind"] == "restart":
        return f
    if case["kind"] == "diagnose":
        return _exact_sums(case, f)
    rho, u = _macros(case, f)
    u[0] += 0.5 * case["force"]
    return rho, u
