"""Performance cases of the framework: what its users have it compute, through its Python API.

A case is a dict of plain values: the flow (``kind``), its lattice and storage, the base grid and block
shape, the refinement levels, and how many coarse steps one pass takes.  A pass of a forward case advances
the simulation by ``steps`` coarse steps (CUDA graphs on a stream of its own, as the benchmark runs it) and
reads back what a program writes out at that point: density and velocity of every level, the level set, and
the observables.  A pass of an adjoint case records ``steps`` steps, and runs the reverse sweep over them.

Inputs are those of the paper's test cases at the sizes of the repository's workloads, tests and benchmark
(``paper_2601_05936_gb300/workloads.py``, ``bench.py``); the seed draws the sub-cell offsets of the bubbles
and interfaces, the surface tension, the densities, viscosities, wall speeds and forces.

Observables and parameter gradients are returned as float32: they are sums over FP32 fields.
"""
import math

import numpy as np
import torch

from paper_2601_05936_gb300 import lsb, workloads

Q_OF = {"D2Q9": 9, "D3Q19": 19, "D3Q27": 27}
FORWARD = ("channel", "couette", "drop", "bubble2d", "bubble3d", "box", "cavity", "ensemble")


def _case(kind, base, steps, levels=1, block=None, storage="fp32", lattice=None, cases=1, radius=0.0, name=None):
    """One case; ``base`` has 2 or 3 entries, ``radius`` is in base cells."""
    D = len(base)
    block = block or ((32, 8) if D == 2 else (32, 4, 4))
    c = dict(kind=kind, lattice=lattice or ("D2Q9" if D == 2 else "D3Q19"), storage=storage, levels=levels, cases=cases,
             nx=base[0], ny=base[1], nz=base[2] if D == 3 else 1, bx=block[0], by=block[1],
             bz=block[2] if D == 3 else 1, radius=float(radius), steps=steps)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # two-layer channel of the validation section: the smallest grid in use, every launch counts
        _case("channel", (64, 32), 20, name="channel2d_64x32"),
        # Laplace test, two levels: small launches, twice per coarse step
        _case("drop", (128, 128), 10, levels=2, radius=20.0, name="drop2d_128x128_L2"),
        # 2D rising bubble on three levels: the level recursion (7 sub-steps a step) and one regrid per pass
        _case("bubble2d", (160, 320), 25, levels=3, radius=40.0, name="bubble2d_160x320_L3"),
        # uneven 2D bubbles of 1-3 levels in one handle (a parameter study), one regrid per pass
        _case("ensemble", (96, 192), 25, levels=3, cases=16, name="ensemble2d_16"),
        # two-layer Couette flow on the large 2D grid, level set live, moving wall: memory-bound 2D
        _case("couette", (2048, 2048), 20, name="couette2d_2048x2048"),
        # single-phase driven box, no-slip walls, odd edges: collide-and-stream alone
        _case("cavity", (250, 251, 253), 20, name="cavity3d_250x251x253"),
        # the benchmark workload: 3D rising bubble on two levels, one regrid per pass
        _case("bubble3d", (128, 128, 256), 25, levels=2, radius=16.0, name="bubble3d_128x128x256_L2"),
        # the same flow with FP16 storage, on a smaller box
        _case("bubble3d", (96, 96, 192), 25, levels=2, radius=12.0, storage="fp16s", name="bubble3d_96x96x192_L2_fp16s"),
        # the paper's own box and lattice: D3Q27, BGK liquid, cumulant gas, slip side walls, uniform grid
        _case("box", (128, 128, 256), 10, lattice="D3Q27", radius=32.0, name="paperbox_d64_D3Q27"),
        # gradients with the level set frozen: reverse sweep over a window of the 3D bubble
        _case("adjoint_frozen", (128, 128, 256), 10, radius=16.0, name="adjoint3d_128x128x256"),
        # gradients through a moving interface, two levels in 2D: many small launches
        _case("adjoint_moving", (64, 96), 8, levels=2, name="adjoint2d_moving_64x96_L2"),
        # the same in 3D: level-set transposes, transfers and the per-call records at size
        _case("adjoint_moving", (96, 96, 128), 4, levels=2, name="adjoint3d_moving_96x96x128_L2"),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(("channel", "couette", "drop", "bubble2d", "ensemble", "cavity", "bubble3d", "bubble3d", "box",
                       "adjoint_frozen", "adjoint_moving"))
    two = rng.choice(((32, 8), (32, 8), (32, 16), (64, 4), (16, 16)))
    three = rng.choice(((32, 4, 4), (32, 4, 4), (16, 8, 4), (64, 4, 2)))
    storage = rng.choice(("fp32", "fp32", "fp16s"))
    if kind == "channel":
        return _case(kind, (log(33, 1024), log(24, 512)), rng.randint(4, 20), block=two, storage=storage)
    if kind == "couette":
        return _case(kind, (log(129, 2048), log(128, 2048)), rng.randint(4, 20), block=two, storage=storage)
    if kind == "drop":
        n = log(64, 192)
        return _case(kind, (n, n + rng.randint(0, 7)), rng.randint(4, 10), levels=rng.randint(1, 3), block=two,
                     radius=n * rng.uniform(0.14, 0.2))
    if kind == "bubble2d":
        w = log(64, 160)
        return _case(kind, (w, 2 * w + rng.randint(-5, 5)), rng.randint(10, 25), levels=rng.randint(1, 3), block=two,
                     storage=storage, radius=w / 4)
    if kind == "ensemble":
        w = log(64, 96)
        return _case(kind, (w, 2 * w), rng.randint(8, 25), levels=rng.randint(1, 3), cases=log(3, 16), block=two)
    if kind == "cavity":
        return _case(kind, (log(40, 250), log(40, 250), log(40, 250)), rng.randint(4, 20), block=three, storage=storage)
    if kind == "bubble3d":
        w = log(40, 120)
        return _case(kind, (w + rng.randint(0, 3), w, 2 * w + rng.randint(0, 5)), rng.randint(4, 25),
                     levels=rng.randint(1, 2), block=three, storage=storage, radius=w / 8)
    if kind == "box":
        d = log(16, 60)
        lattice = rng.choice(("D3Q19", "D3Q27"))
        return _case(kind, (2 * d, 2 * d, 4 * d), rng.randint(4, 10), block=(32, 4, 4), lattice=lattice, radius=d / 2)
    if kind == "adjoint_frozen":
        w = log(32, 120)
        return _case(kind, (w, w + rng.randint(0, 3), 2 * w), rng.randint(3, 8), levels=1 if w > 48 else rng.randint(1, 2),
                     block=three, radius=w / 8)
    if rng.random() < 0.5:
        return _case(kind, (log(33, 160), log(48, 160)), rng.randint(3, 8), levels=rng.randint(1, 2), block=two)
    return _case(kind, (log(24, 88), log(24, 88), log(32, 112)), rng.randint(2, 4), levels=rng.randint(1, 2))


# ------------------------------------------------------------------ inputs
def _dims(c):
    return (c["nx"], c["ny"]) if c["lattice"] == "D2Q9" else (c["nx"], c["ny"], c["nz"])


def _centres(dims):
    """Cell-centre coordinates on the GPU, broadcastable, in the order of the axes (x is the last dimension)."""
    D = len(dims)
    return [(torch.arange(n, dtype=torch.float64, device="cuda") + 0.5).reshape([-1 if D - 1 - k == a else 1 for k in range(D)])
            for a, n in enumerate(dims)]


def _ball(dims, centre, R):
    return R - torch.sqrt(sum((x - p) ** 2 for x, p in zip(_centres(dims), centre)))


def _host(phi):
    return phi.to(torch.float32).reshape(-1).cpu().numpy()


def _layered_flow(c, rng):
    """The two-layer channel (body force) and Couette (moving top wall) flows: periodic in x, flat interface."""
    ny, couette = c["ny"], c["kind"] == "couette"
    rho, eta_ratio = (1.0, 0.1), 5.0
    nu_l = 0.1 * rng.uniform(0.9, 1.1)
    h = math.floor(0.5 * ny) + rng.uniform(0.1, 0.9) + 0.5
    y = _centres(_dims(c))[1]
    phi = (y - h).expand(ny, c["nx"])
    wall = np.zeros((4, 2))
    force = 0.0
    if couette:
        wall[3, 0] = 0.01 * rng.uniform(0.9, 1.1)
    else:
        force = 8.0 * nu_l * 0.01 * rng.uniform(0.9, 1.1) / ny ** 2
    return dict(periodic=(True, False), rho_phys=rho, nu=(nu_l, nu_l * rho[0] / eta_ratio / rho[1]), sigma=0.0,
                body_force=(force, 0.0), wall_u=wall.reshape(-1), phi0=_host(phi))


def _drop(c, rng):
    """Static gas bubble in a periodic box of liquid, density ratio 1000."""
    r = 2 ** (c["levels"] - 1)
    nf = tuple(n * r for n in _dims(c))
    sigma, R = rng.uniform(1e-3, 1e-2), c["radius"] * r
    centre = [n / 2 + rng.random() * r for n in nf]
    return dict(periodic=(True, True), rho_phys=(1.0, 1e-3), nu=(0.1, 1.0), sigma=sigma, p_gas0=sigma / R,
                phi0=_host(_ball(nf, centre, R)), refine_dist=[4.0] * (c["levels"] - 1), sensor="band", regrid_every=0)


def _bubble(c, rng, frozen=False):
    """Rising bubble in a no-slip box at 1/4 height: density ratio 1000, viscosity ratio 100; with FP16 storage the
    paper's parameter set I (both 10), members of an ensemble in between."""
    base, L = _dims(c), c["levels"]
    D, r = len(base), 2 ** (c["levels"] - 1)
    nf = tuple(n * r for n in base)
    R = c["radius"] * r
    ratios = (1000.0, 100.0) if c["storage"] == "fp32" else (10.0, 10.0)
    if c["kind"] == "ensemble":
        ratios = (10.0 ** rng.uniform(1.0, 2.0), 10.0)
    prm = workloads.bubble_params(2 * R, 35.0, 10.0 * rng.uniform(0.8, 1.2), *ratios, Ma=0.005)
    centre = [(n / 2 if a < D - 1 else n / 4) * r + rng.random() * 0.5 * r for a, n in enumerate(base)]
    dist = 16.0 if D == 2 else max(8.0, 2.0 * c["radius"])
    dref = [48.0] + [16.0] * (L - 2) if L > 2 else [dist] * (L - 1)
    grav = (0.0,) * (D - 1) + (-prm["g"],)
    p = dict(periodic=(False,) * D, rho_phys=prm["rho_phys"], nu=prm["nu"], gravity=grav, sigma=prm["sigma"],
             x_ref=centre, p_gas0=(D - 1) * prm["sigma"] / R, phi0=_host(_ball(nf, centre, R)), refine_dist=dref,
             sensor="band", regrid_every=25)
    if frozen:
        p.update(ls_active=False, n_ext=0, reinit_every=0, regrid_every=0)
    return p


def _paper_box(c, rng):
    """The paper's 2d x 2d x 4d box, parameter set I, slip side walls; on D3Q27 the gas takes the cumulant model."""
    d = 2.0 * c["radius"]
    prm = workloads.bubble_params(d, Ma=0.005, nu_floor=0.1, **workloads.PAPER_CASES["I"])
    centre = [d + rng.random() * 0.5 for _ in range(3)]
    return dict(periodic=(False,) * 3, slip=(True, True, False), rho_phys=prm["rho_phys"], nu=prm["nu"],
                gravity=(0.0, 0.0, -prm["g"]), sigma=prm["sigma"], x_ref=centre, p_gas0=2.0 * prm["sigma"] / (d / 2),
                phi0=_host(_ball(_dims(c), centre, d / 2)), collision=("bgk", "cumulant" if c["lattice"] == "D3Q27" else "bgk"))


def _cavity(c, rng):
    """Liquid in a box whose six walls slide in their own planes, with a body force."""
    wall = rng.uniform(-0.02, 0.02, (6, 3))
    for f in range(6):
        wall[f, f // 2] = 0.0
    nu = rng.uniform(0.03, 0.06)
    return dict(periodic=(False,) * 3, rho_phys=(1.0, 1.0), nu=(nu, nu), body_force=tuple(rng.uniform(-1e-6, 1e-6, 3)),
                wall_u=wall.reshape(-1), phi0=-np.ones(c["nx"] * c["ny"] * c["nz"], np.float32), ls_active=False, n_ext=0,
                reinit_every=0)


def _wavy_layer(c, rng):
    """Liquid below gas with a gently wavy interface that passes between two layers of cell centres, so that no
    cell changes phase while it relaxes (the adjoint's condition); a sliding lid drives the flow."""
    r = 2 ** (c["levels"] - 1)
    nf = tuple(n * r for n in _dims(c))
    D = len(nf)
    X = _centres(nf)
    h = nf[D - 1] // 2 + 1.0 + rng.uniform(-0.05, 0.05)
    wave = 0.12 * torch.sin(2 * math.pi * X[0] / nf[0] + rng.uniform(0, 6.28))
    if D == 3:
        wave = wave + 0.08 * torch.sin(2 * math.pi * X[1] / nf[1] + rng.uniform(0, 6.28))
    wall = np.zeros((2 * D, D))
    wall[2 * D - 1, 0] = 0.005 * rng.uniform(0.8, 1.2)
    return dict(periodic=(True,) * (D - 1) + (False,), rho_phys=(1.0, 0.1), nu=(0.08, 0.3), sigma=0.002 * rng.uniform(0.8, 1.2),
                body_force=(1e-6,) + (0.0,) * (D - 1), wall_u=wall.reshape(-1),
                phi0=_host((X[D - 1] - h - wave).expand(nf[::-1])), refine_dist=[6.0] * (c["levels"] - 1), sensor="band",
                regrid_every=0)


def _descriptions(c, seed):
    """The library's case dictionaries of one handle."""
    out = []
    for k in range(c["cases"]):
        rng = np.random.default_rng([seed, k])
        own = dict(c)
        if c["kind"] == "ensemble":  # uneven members: width, levels and radius their own (the same for every seed)
            size = np.random.default_rng([c["nx"], k])
            w = 2 * int(size.integers(c["nx"] // 2, c["nx"] + 1))
            own.update(nx=w, ny=2 * w, levels=1 + k % c["levels"], radius=w / 8.0)
        make = dict(channel=_layered_flow, couette=_layered_flow, drop=_drop, bubble2d=_bubble, bubble3d=_bubble, ensemble=_bubble,
                    box=_paper_box, cavity=_cavity, adjoint_moving=_wavy_layer,
                    adjoint_frozen=lambda a, b: _bubble(a, b, frozen=True))[c["kind"]]
        D = 2 if c["lattice"] == "D2Q9" else 3
        out.append({**workloads.LS_DEFAULTS, "name": c["kind"], "lattice": c["lattice"], "base": _dims(own),
                    "block": (c["bx"], c["by"], c["bz"])[:D], "n_levels": own["levels"], "storage": c["storage"],
                    "fp16_scale": 1024.0, **make(own, rng)})
    return out


# ------------------------------------------------------------------ the cases' passes
def prepare(case, seed):
    """The handle a program keeps, and the device arrays it reads the fields into."""
    cases = _descriptions(case, seed)
    grid = lsb.Grid(cases, stream=torch.cuda.Stream())
    if case["kind"] in FORWARD:
        grid.use_graphs(True)
    read = []  # (case, level, field, array)
    for k, c in enumerate(cases):
        D, L = len(c["base"]), c["n_levels"]
        for l in range(L):
            shape = tuple(n * 2 ** l for n in c["base"])[::-1]
            read.append((k, l, "rho", shape))
            read.append((k, l, "u", (D,) + shape))
        if c["ls_active"] if "ls_active" in c else True:
            read.append((k, L - 1, "phi", shape))
    # one array per field, the cases' and levels' dense boxes one after the other
    sizes = {f: sum(math.prod(s) for _, _, g, s in read if g == f) for f in ("rho", "u", "phi")}
    arrays = {f: torch.zeros(n, dtype=torch.float32, device="cuda") for f, n in sizes.items() if n}
    at = dict.fromkeys(arrays, 0)
    fields = []
    for k, l, f, s in read:
        n = math.prod(s)
        fields.append((k, l, f, arrays[f][at[f]:at[f] + n]))
        at[f] += n
    weights = np.zeros((len(cases), 4 + 2 * grid.D))
    weights[:, 0] = 1e-3                  # liquid mass
    weights[:, 3 + 2 * grid.D] = 1.0      # gas velocity along the last axis
    weights[:, 4 + grid.D] = 0.5          # ... and along x
    return dict(case=case, grid=grid, fields=fields, arrays=arrays, weights=weights)


def run(state):
    g, case = state["grid"], state["case"]
    out = dict(state["arrays"])
    if case["kind"] in FORWARD:
        g.step(case["steps"])
        if case["kind"] != "cavity":  # (no gas in it)
            obs = g.observables()
            out["observables"] = np.array([[*o["mass"], o["volume"], *o["centroid"], *o["velocity"]] for o in obs], np.float32)
    else:
        g.record(case["steps"])
        g.step(case["steps"])
        dp, dphi = g.backward(state["weights"], want_phi=True)
        out["dparams"] = dp.astype(np.float32)
        out["dphi"] = [d for d in dphi]
    for k, l, field, a in state["fields"]:
        g.get_device(field, a.data_ptr(), a.numel() * 4, case_idx=k, level=l)
    return out


def _cells(case):
    """Per member of the handle: cells of its level boxes and a rough count of the leaves and of the band."""
    out = []
    for k in range(case["cases"]):
        own = dict(case)
        if case["kind"] == "ensemble":
            size = np.random.default_rng([case["nx"], k])
            w = 2 * int(size.integers(case["nx"] // 2, case["nx"] + 1))
            own.update(nx=w, ny=2 * w, levels=1 + k % case["levels"], radius=w / 8.0)
        base = _dims(own)
        D, L = len(base), own["levels"]
        box = [math.prod(base) * 2 ** (D * l) for l in range(L)]
        top = [n * 2 ** (L - 1) for n in base]
        if case["kind"] == "cavity":
            surface = 0.0
        elif case["kind"] in ("channel", "couette", "adjoint_moving"):
            surface = float(math.prod(top[:-1]))
        else:
            R = own["radius"] * 2 ** (L - 1)
            surface = 2 * math.pi * R if D == 2 else 4 * math.pi * R * R
        # refined: the cells within the refinement distance of the interface (in finest cells; three times that on
        # the coarser levels of three); the rest of each box is a leaf of the level above
        reach = {"drop": 4.0, "adjoint_moving": 6.0}.get(case["kind"], 16.0 if D == 2 else max(8.0, 2.0 * own["radius"]))
        updates, covered = 0.0, 0.0
        for l in reversed(range(L)):
            r = 2 ** (L - 1 - l)
            active = box[l] if l == 0 else min(box[l], surface * 2 * reach * (3 if l < L - 1 else 1) / r ** D)
            updates += max(0.0, active - covered / 2 ** D) * 2 ** l
            covered = active
        out.append(dict(D=D, box=box, updates=updates, surface=surface * 2 ** (L - 1)))
    return out


def work(case):
    """Per coarse step: every leaf's populations read and written once; in the band (about 8 cells on both sides
    of the interface) phi and the extension velocity read and written once; fields written once per pass."""
    Q, es = Q_OF[case["lattice"]], 2 if case["storage"] == "fp16s" else 4
    bytes_, flops = 0.0, 0.0
    for m in _cells(case):
        D, n = m["D"], case["steps"]
        moving = case["kind"] not in ("cavity", "adjoint_frozen")
        band = 16.0 * m["surface"] * 2 * 4 * (1 + D) if moving else 0.0
        step = 2.0 * Q * es * m["updates"] + band
        ops = (12.0 * Q + 30) * m["updates"] + (16.0 * m["surface"] * (8 * 12 * D + 3 * 20 * D + 3 * 120 * D) if moving else 0.0)
        if case["kind"] in FORWARD:
            fields = 4.0 * (1 + D) * sum(m["box"]) + (4.0 * m["box"][-1] if moving else 0.0)
            bytes_ += n * step + fields
            flops += n * ops
        else:
            # forward twice (recorded, recomputed), then the adjoint step: state and adjoint read, adjoint written
            bytes_ += n * (2 * step + 1.5 * step) + 4.0 * (2 + D) * sum(m["box"])
            flops += n * 5 * ops
    return dict(bytes=bytes_, flops=flops)


# ------------------------------------------------------------------ the same in 64 bits
_D2Q9 = [(-1, 0), (1, 0), (0, -1), (0, 1), (-1, -1), (-1, 1), (1, 1), (1, -1), (0, 0)]
_D3Q19 = [(-1, 0, 0), (1, 0, 0), (0, -1, 0), (0, 1, 0), (0, 0, -1), (0, 0, 1), (-1, -1, 0), (-1, 1, 0), (1, -1, 0), (1, 1, 0),
          (-1, 0, -1), (-1, 0, 1), (1, 0, -1), (1, 0, 1), (0, -1, -1), (0, -1, 1), (0, 1, -1), (0, 1, 1), (0, 0, 0)]


def _weights(c):
    D = len(c[0])
    by = {2: {0: 4 / 9, 1: 1 / 9, 2: 1 / 36}, 3: {0: 1 / 3, 1: 1 / 18, 2: 1 / 36}}[D]
    return [by[sum(abs(a) for a in v)] for v in c]


def _bgk(f, c, w, omega, acc):
    """Post-collision deviations f - w, with the moments (Eqs. 1, feq, forcing)."""
    D = len(c[0])
    drho = sum(f)
    rho = 1 + drho
    u = [sum(v[a] * fi for v, fi in zip(c, f) if v[a]) / rho for a in range(D)]
    usq = sum(x * x for x in u)
    out = []
    for v, wi, fi in zip(c, w, f):
        cu = sum(v[a] * u[a] for a in range(D))
        ca = sum(v[a] * acc[a] for a in range(D))
        eq = wi * (drho + rho * (3 * cu + 4.5 * cu * cu - 1.5 * usq))
        out.append(fi + omega * (eq - fi) + 3 * wi * rho * ca)
    return out, rho, u


def _exact_cavity(case, p):
    c, w = _D3Q19, _weights(_D3Q19)
    shape = (case["nz"], case["ny"], case["nx"])
    opp = [c.index(tuple(-a for a in v)) for v in c]
    wall = np.asarray(p["wall_u"]).reshape(6, 3)
    f = [torch.zeros(shape, dtype=torch.float64, device="cuda") for _ in c]
    omega = 1.0 / (3.0 * p["nu"][0] + 0.5)
    for _ in range(case["steps"]):
        f, _, _ = _bgk(f, c, w, omega, p["body_force"])
        new = [None] * len(c)
        for i, v in enumerate(c):  # population i of x goes to x + c_i, or back from the wall it meets
            g = torch.empty_like(f[i])
            g.copy_(f[opp[i]])     # what bounced back into i at x left x along opp(i)
            for a in reversed(range(3)):  # where several walls meet, the one of the first axis counts
                if v[a]:
                    face = 2 * a + (0 if v[a] > 0 else 1)  # direction opp(i) points at this wall
                    at = [slice(None)] * 3
                    at[2 - a] = 0 if v[a] > 0 else -1
                    du = -sum(v[b] * wall[face, b] for b in range(3))
                    g[tuple(at)] = f[opp[i]][tuple(at)] - 6 * w[i] * du
            src, dst = [slice(None)] * 3, [slice(None)] * 3
            for a in range(3):
                if v[a] > 0:
                    src[2 - a], dst[2 - a] = slice(None, -1), slice(1, None)
                elif v[a] < 0:
                    src[2 - a], dst[2 - a] = slice(1, None), slice(None, -1)
            g[tuple(dst)] = f[i][tuple(src)]
            new[i] = g
        f = new
    _, rho, u = _bgk(f, c, w, omega, p["body_force"])
    return dict(rho=rho.reshape(-1), u=torch.stack(u).reshape(-1))


def _exact_layers(case, p):
    """The layered flows are uniform in x and their interface stays put: one column of cells, both phases."""
    c, w = _D2Q9, _weights(_D2Q9)
    opp = [c.index((-a, -b)) for a, b in c]
    ny, n = case["ny"], case["nx"]
    phi = p["phi0"].reshape(ny, n)[:, 0].astype(np.float64)
    gas = (phi >= 0).astype(int)
    rho_k, nu = np.asarray(p["rho_phys"]), np.asarray(p["nu"])
    omega, acc, eta = 1 / (3 * nu + 0.5), [[p["body_force"][0] / r, 0.0] for r in rho_k], rho_k * nu
    wall = np.asarray(p["wall_u"]).reshape(4, 2)
    j = int(np.argmax(gas))  # first gas row; the cut links run between rows j - 1 and j
    f = [np.zeros(ny) for _ in c]
    om = omega[gas]
    for _ in range(case["steps"]):
        pre = f
        f, rho, u = _bgk(f, c, w, om, [np.asarray([a[b] for a in acc])[gas] for b in range(2)])
        drho, usq = rho - 1, u[0] ** 2 + u[1] ** 2
        S = np.zeros((2, 2, ny))
        for v, wi, fi in zip(c, w, pre):
            cu = v[0] * u[0] + v[1] * u[1]
            neq = fi - wi * (drho + rho * (3 * cu + 4.5 * cu * cu - 1.5 * usq))
            for a in range(2):
                for b in range(2):
                    S[a, b] -= 1.5 * om / rho * v[a] * v[b] * neq
        new = [np.empty(ny) for _ in c]
        for i, v in enumerate(c):
            s = v[1]
            if s == 0:
                new[i][:] = f[i]
                continue
            if s > 0:
                new[i][1:] = f[i][:-1]
            else:
                new[i][:-1] = f[i][1:]
            face, row = (2, 0) if s > 0 else (3, ny - 1)
            o = opp[i]
            new[i][row] = f[o][row] - 6 * w[i] * (c[o][0] * wall[face, 0] + c[o][1] * wall[face, 1])
        for x, y, A in ((j - 1, j, 0), (j, j - 1, 1)):  # cell x of phase A, its partner y
            q = phi[x] / (phi[x] - phi[y])
            sgn = 1.0 if A == 0 else -1.0
            nv = np.array([0.0, sgn])
            uI = np.array([(1 - q) * u[a][x] + q * u[a][y] for a in range(2)])
            Sb = 0.5 * (S[:, :, x] + S[:, :, y])
            jp = (rho_k[1 - A] * drho[y] - rho_k[A] * drho[x]) / 3
            eb, je = 0.5 * (eta[0] + eta[1]), eta[1 - A] - eta[A]
            v_ = Sb @ nv
            Snn = nv @ v_
            vt = v_ - Snn * nv
            for i, ci in enumerate(c):
                if ci[1] != y - x:
                    continue
                k = opp[i]
                cn, cvt = np.dot(ci, nv), np.dot(ci, vt)
                ccS = (jp / (2 * eb) - je / eb * Snn) * cn * cn - 2 * je / eb * cn * cvt
                df = -6 * w[i] * (np.dot(ci, uI) - q * (1 - q) * ccS)
                if q >= 0.5:
                    new[k][x] = f[i][x] / (2 * q) + (2 * q - 1) / (2 * q) * f[k][x] + df / (2 * q)
                else:
                    new[k][x] = 2 * q * f[i][x] + (1 - 2 * q) * new[i][x] + df
        f = new
    _, rho, u = _bgk(f, c, w, om, [0.0, 0.0])

    def wide(v):
        return np.repeat(np.asarray(v, np.float64).reshape(-1, 1), n, axis=1).reshape(-1)

    return dict(rho=wide(rho), u=np.concatenate([wide(u[0]), wide(u[1])]), phi=p["phi0"].astype(np.float64),
                observables=None)


def exact(case, seed):
    """Single-phase boxes and the layered two-phase flows (FP32 storage); the curved, moving interfaces, the level
    transfers and the reverse sweeps have no short plain form."""
    if case["storage"] != "fp32" or case["kind"] not in ("cavity", "channel", "couette"):
        return None
    p = _descriptions(case, seed)[0]
    return _exact_cavity(case, p) if case["kind"] == "cavity" else _exact_layers(case, p)
