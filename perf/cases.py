"""What a user of this framework has it do, as cases that can be timed: whole passes through the
public entry points (Sim, lbm_init, lbm_step, lbm_moments_async, lbm_conserved, lbm_get_state,
lbm_batch_step) on grids from a few hundred sites to tens of millions, both lattices, every storage
format, every kind of wall and force.

A case is a dict of plain values:
  flow       the problem, which fixes walls and force (FLOWS below)
  lattice    "D2Q37" or "D3Q39"; nx, ny, nz the grid
  storage    "fp64" (IEEE double), "fp64_pair" (FP64 storage, float-float step), "fp32", "fp16"
  order      force order 0, 1, 2; tau the relaxation time (unused by the constant-viscosity flows)
  use        "simulate": fields in, steps, fields out; "advance": steps, fields out, the state goes
             on; "monitor": fields in, after every step the conserved sums, fields out;
             "checkpoint": as "advance" and the populations out; "batch": many grids per launch
  steps      steps of one pass; graph_steps: steps per replayed graph
  count      grids of a batch
Inputs are made on the GPU from the seed: the flow's mean fields, a few smooth modes of velocity,
density and temperature with random phases (the convection rolls, jets and waves that such runs
develop) and a little noise.
"""
import math

import numpy as np
import torch

import paper_2302_04741_gb300 as lbm

PRECISION = {"fp64": lbm.LBM_FP64, "fp64_pair": lbm.LBM_FP64, "fp32": lbm.LBM_FP32_SHIFTED,
             "fp16": lbm.LBM_FP16_SCALED}
BYTES = {"fp64": 8, "fp64_pair": 8, "fp32": 4, "fp16": 2}
# walls of the last axis, and the kind of force, of each flow
FLOWS = {"kolmogorov": ("periodic", "sine"), "convection": ("thermal", "uniform"),
         "poiseuille": ("thermal", "uniform"), "channel": ("bounce", "uniform"),
         "box": ("periodic", "uniform"), "cylinders": ("periodic", "field")}
WALL = {"periodic": 0, "bounce": 1, "thermal": 2}
SIDES = (128, 192, 256, 384, 512)  # of the grids of a batch


def listed():
    two, three = {"lattice": "D2Q37", "nz": 1}, {"lattice": "D3Q39"}
    return [
        # The compressible Poiseuille validation: 450 sites, hundreds of thousands of steps, so the
        # latency of a step is everything. Constant viscosity, hot and cold wall.
        dict(two, name="poiseuille_3x150_fp64", flow="poiseuille", nx=3, ny=150, storage="fp64", order=2, tau=1.0,
             use="advance", steps=200, graph_steps=100),
        # The periodic accuracy problem at its usual size, in double, with its populations.
        dict(two, name="kolmogorov_64x64_fp64", flow="kolmogorov", nx=64, ny=64, storage="fp64", order=2, tau=0.8,
             use="checkpoint", steps=100, graph_steps=10),
        # Rotating concentric cylinders: a staircase of solid sites, a force field, constant viscosity.
        dict(two, name="cylinders_256x256_fp64", flow="cylinders", nx=256, ny=256, storage="fp64", order=2, tau=1.0,
             use="advance", steps=20, graph_steps=10),
        # A small run that is watched: conserved sums on the host after every step.
        dict(two, name="monitor_300x100_fp32", flow="convection", nx=300, ny=100, storage="fp32", order=2, tau=0.6,
             use="monitor", steps=10, graph_steps=0),
        # The benchmark's convection cell, 50 steps, then the fields.
        dict(two, name="convection_1024x512_fp32", flow="convection", nx=1024, ny=512, storage="fp32", order=2, tau=0.6,
             use="advance", steps=50, graph_steps=50),
        # The same cell in double, the default storage and arithmetic, checkpointed.
        dict(two, name="convection_1024x512_fp64", flow="convection", nx=1024, ny=512, storage="fp64", order=2, tau=0.6,
             use="checkpoint", steps=10, graph_steps=10),
        # The same cell with float-float arithmetic, the fast way to FP64 accuracy.
        dict(two, name="convection_1024x512_pair", flow="convection", nx=1024, ny=512, storage="fp64_pair", order=2,
             tau=0.6, use="advance", steps=10, graph_steps=10),
        # An odd-sized channel between no-slip walls in half storage, the Guo force, from its fields.
        dict(two, name="channel_1021x509_fp16", flow="channel", nx=1021, ny=509, storage="fp16", order=1, tau=0.7,
             use="simulate", steps=50, graph_steps=10),
        # A parameter study: 64 independent grids of mixed sizes stepped by one launch.
        dict(two, name="batch_64_fp32", flow="kolmogorov", nx=0, ny=0, storage="fp32", order=2, tau=0.8, use="batch",
             steps=20, graph_steps=10, count=64),
        # One request of the 3-D service: fields in, steps, fields out.
        dict(three, name="box_96_fp32", flow="box", nx=96, ny=96, nz=96, storage="fp32", order=2, tau=0.8,
             use="simulate", steps=50, graph_steps=10),
        # A small 3-D reference run in double on an odd grid.
        dict(three, name="box_61x47x53_fp64", flow="box", nx=61, ny=47, nz=53, storage="fp64", order=2, tau=0.8,
             use="simulate", steps=20, graph_steps=10),
        # The large 3-D convection cell in half storage: 67 million sites.
        dict(three, name="convection_512x512x256_fp16", flow="convection", nx=512, ny=512, nz=256, storage="fp16",
             order=2, tau=0.55, use="advance", steps=20, graph_steps=0),
    ]


# time of a site and step in picoseconds, to bound a drawn case's cost
COST = {"fp64": 1250.0, "fp64_pair": 500.0, "fp32": 60.0, "fp16": 60.0}


def draw(rng):
    """A case of one of the families above, sizes spread over their ranges' logarithm."""
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    family = rng.choice(("plane", "plane", "plane", "space", "space", "batch", "cylinders", "monitor", "large"))
    c = {"order": rng.choice((0, 1, 2, 2, 2)), "tau": round(rng.uniform(0.55, 1.0), 3),
         "graph_steps": rng.choice((0, 2, 10, 10))}
    if family == "batch":
        c.update(lattice="D2Q37", nz=1, flow="kolmogorov", nx=0, ny=0, storage=rng.choice(("fp32", "fp32", "fp16")),
                 use="batch", count=size(2, 64))
    elif family == "cylinders":
        n = size(40, 256)
        c.update(lattice="D2Q37", nz=1, flow="cylinders", nx=n, ny=n, storage=rng.choice(("fp64", "fp32")), use="advance")
    elif family == "large":
        c.update(lattice="D3Q39", flow=rng.choice(("convection", "box", "channel")), nx=size(129, 500), ny=size(129, 500),
                 nz=size(65, 250), storage=rng.choice(("fp32", "fp16", "fp16")), use="advance")
    elif family == "space":
        c.update(lattice="D3Q39", flow=rng.choice(("box", "box", "convection", "kolmogorov")), nx=size(24, 128),
                 ny=size(24, 128), nz=size(24, 128), storage=rng.choice(("fp64", "fp64_pair", "fp32", "fp32", "fp16")),
                 use=rng.choice(("simulate", "advance")))
    else:
        c.update(lattice="D2Q37", nz=1, flow=rng.choice(("kolmogorov", "convection", "channel", "poiseuille")),
                 nx=size(16, 1500), ny=size(24, 700), storage=rng.choice(("fp64", "fp64", "fp64_pair", "fp32", "fp16")),
                 use=rng.choice(("simulate", "advance", "checkpoint")))
        if family == "monitor":
            c.update(use="monitor", storage=rng.choice(("fp64", "fp32")), graph_steps=0)
            c["nx"], c["ny"] = min(c["nx"], 600), min(c["ny"], 300)
        if c["flow"] == "poiseuille":
            c.update(nx=rng.choice((3, 4, 7, 33)), ny=size(40, 300), storage="fp64", use="advance")
    sites = c["nx"] * c["ny"] * c["nz"] if c["use"] != "batch" else 80000 * c["count"]
    step_s = max(5e-6, sites * COST[c["storage"]] * 1e-12)
    most = int(max(2, min(200, 0.02 / step_s)))
    c["steps"] = size(2, most) if c["use"] != "monitor" else size(2, 12)
    return c


def dims(case):
    return 2 if case["lattice"] == "D2Q37" else 3


def grids(case, seed):
    """(nx, ny, nz, tau, g0) of every grid of the case."""
    if case["use"] != "batch":
        return [(case["nx"], case["ny"], case["nz"], case["tau"], 1e-5)]
    r = np.random.RandomState(case["count"])  # the mix belongs to the case, the values to the seed
    shapes = [(int(r.choice(SIDES)), int(r.choice(SIDES))) for _ in range(case["count"])]
    v = np.random.RandomState(seed % (1 << 31))
    return [(nx, ny, 1, float(v.uniform(0.55, 1.0)), float(10.0 ** v.uniform(-6, -4))) for nx, ny in shapes]


def problem(case, grid, seed):
    """Parameters (host values) and fields (float64, on the GPU) of one grid: what a program hands to lbm_create and
    lbm_init."""
    nx, ny, nz, tau, g0 = grid
    D, N = dims(case), nx * ny * nz
    flow = case["flow"]
    wall, force = FLOWS[flow]
    gen = torch.Generator(device="cuda").manual_seed(int(seed) & 0x7FFFFFFF)

    def rand(n, a, b):
        return a + (b - a) * torch.rand(n, generator=gen, dtype=torch.float64, device="cuda")

    x = torch.arange(nx, dtype=torch.float64, device="cuda").view(1, 1, nx)
    y = torch.arange(ny, dtype=torch.float64, device="cuda").view(1, ny, 1)
    z = torch.arange(nz, dtype=torch.float64, device="cuda").view(nz, 1, 1)
    n_wall = ny if D == 2 else nz
    s = ((y if D == 2 else z) + 0.5) / n_wall  # 0..1 across the last axis
    ph = rand(8, 0.0, 2.0 * math.pi)
    kx, ky, kz = 2.0 * math.pi * x / nx, 2.0 * math.pi * y / ny, 2.0 * math.pi * z / nz
    p = dict(D=D, shape=(nx, ny, nz), N=N, tau=tau, mu=0.0, wall=wall, T_lo=1.0, T_hi=1.0, g={"kind": lbm.LBM_G_UNIFORM,
             "g0": (0.0, 0.0, 0.0)}, solid=None, T_wall=None)
    down = [0.0, 0.0, 0.0]
    if force == "sine":
        p["g"] = {"kind": lbm.LBM_G_SINE, "g0": (g0, 0.0, 0.0), "wave_axis": 1}
        T, flow_u = 1.0 + 0.01 * torch.sin(kx + ph[0]) + 0.0 * (ky + kz), 0.02
    elif flow == "convection":
        p["T_lo"], p["T_hi"] = 1.05, 0.95
        down[D - 1] = -g0
        T, flow_u = p["T_lo"] + (p["T_hi"] - p["T_lo"]) * s + 0.0 * (kx + ky + kz), 0.02
    elif flow == "poiseuille":  # g_x = 8 mu U / H^2 and g_y = -50 g_x; at the height of 150 the paper's first case (U =
        # 1.5, Re = 1800), lower channels at the same viscosity and a Mach number in proportion
        H, U = ny * 1.196979770393, 1.5 * min(1.0, ny / 150.0)
        p["mu"] = 1.5 * 150 * 1.196979770393 / 1800.0
        gx = 8.0 * p["mu"] * U / (H * H)
        p["T_lo"], p["T_hi"] = 1.0, 1.1
        down = [gx, -50.0 * gx, 0.0]
        T, flow_u = 1.0 + 0.1 * s + 0.0 * kx, 0.0
    elif flow == "channel":
        down[0] = g0
        T, flow_u = 1.0 + 0.02 * torch.cos(kx + ph[0]) + 0.0 * (ky + kz), 0.02
    elif flow == "box":
        down[D - 1] = -g0
        T, flow_u = 1.0 + 0.01 * torch.sin(kx + ph[0]) * torch.cos(kz + ph[1]) + 0.0 * ky, 0.02
    else:  # cylinders of radii R and R / 5 in the co-rotating frame, Re = 100, centre-line speed 0.3
        Ro = (nx - 6) * 1.196979770393 / 2.0
        Ri = Ro / 5.0
        alpha = 0.3 / (0.5 * (Ro + Ri))
        p["mu"] = alpha * (Ro * Ro - Ri * Ri) / 200.0
        X, Y = 1.196979770393 * (x - 0.5 * (nx - 1)), 1.196979770393 * (y - 0.5 * (ny - 1))
        X, Y = (X + 0.0 * Y), (Y + 0.0 * X)
        R = torch.hypot(X, Y)
        inner, outer = R < Ri, R > Ro
        p["solid"] = (inner | outer).reshape(N).to(torch.uint8).cpu().numpy()
        p["T_wall"] = torch.where(inner, 1.0, 1.1).double().reshape(N).cpu().numpy()
        p["g"] = {"kind": lbm.LBM_G_FIELD, "field": torch.stack([alpha ** 2 * X, alpha ** 2 * Y]).reshape(2, N).contiguous()}
        T, flow_u = 1.0 + 0.1 * torch.log(R.clamp(Ri, Ro) / Ri) / math.log(5.0), 0.0
    if force == "uniform":
        p["g"]["g0"] = tuple(down)
    T = (T.expand(nz, ny, nx).reshape(N) + rand(N, -1e-4, 1e-4)).contiguous()
    rho = 1.0 + 1e-3 * torch.cos(kx + ph[2]) * torch.cos((ky if D == 2 else kz) + ph[3]) + 0.0 * (ky + kz)
    if flow == "cylinders":
        rho = 1.0 + 0.0 * R
    rho = (rho.expand(nz, ny, nx).reshape(N) + rand(N, -1e-6, 1e-6)).contiguous()
    u = torch.zeros(D, N, dtype=torch.float64, device="cuda")
    if flow_u:  # rolls: along x with the shape of the last axis, and back across it
        across = torch.sin(math.pi * s) if wall != "periodic" else torch.sin((ky if D == 2 else kz) + ph[4])
        u[0] = (flow_u * torch.cos(kx + ph[5]) * across + 0.0 * (ky + kz)).reshape(N)
        u[D - 1] = (flow_u * torch.sin(kx + ph[6]) * across + 0.0 * (ky + kz)).reshape(N)
        if D == 3:
            u[1] = (0.5 * flow_u * torch.sin(ky + ph[7]) * across + 0.0 * kx).reshape(N)
    elif flow == "poiseuille":  # towards its parabola
        u[0] = (2.0 * U * s * (1.0 - s) + 0.0 * kx).reshape(N)
    p["rho"], p["u"], p["T"] = rho, u, T
    return p


def prepare(case, seed):
    D, lat = dims(case), lbm.LBM_D2Q37 if case["lattice"] == "D2Q37" else lbm.LBM_D3Q39
    batch = case["use"] == "batch"
    stream = torch.cuda.Stream() if batch else None
    members = []
    mine = grids(case, seed)
    total = sum(nx * ny * nz for nx, ny, nz, _, _ in mine)
    out = {k: torch.zeros(n * total, dtype=torch.float64, device="cuda") for k, n in (("rho", 1), ("u", D), ("T", 1), ("q", D))}
    at = 0
    for k, grid in enumerate(mine):
        p = problem(case, grid, seed * 1009 + k)
        nx, ny, nz = p["shape"]
        bc, T_lo, T_hi = [0, 0, 0], [1.0] * 3, [1.0] * 3
        bc[D - 1], T_lo[D - 1], T_hi[D - 1] = WALL[p["wall"]], p["T_lo"], p["T_hi"]
        w = dict(lattice=lat, shape=(nx, ny, nz), tau=p["tau"], mu=p["mu"], precision=PRECISION[case["storage"]],
                 force_order=case["order"], bc=tuple(bc), T_lo=tuple(T_lo), T_hi=tuple(T_hi), g=p["g"],
                 fp64_arith=int(case["storage"] == "fp64_pair"), rho=p["rho"], u=p["u"], T=p["T"])
        if p["solid"] is not None:
            w["solid"], w["T_wall"] = p["solid"], p["T_wall"]
        torch.cuda.synchronize()
        sim = lbm.Sim(w, stream=stream.cuda_stream if batch else None, graph_steps=0 if batch else case["graph_steps"]).init()
        N = p["N"]
        members.append((sim, out["rho"][at:at + N], out["u"][D * at:D * (at + N)], out["T"][at:at + N],
                        out["q"][D * at:D * (at + N)]))
        at += N
    state = dict(case=case, sims=members, out=out, stream=stream, batch=None)
    if batch:
        state["batch"] = Batch(lat, case, stream, [m[0] for m in members])
    if case["use"] == "checkpoint":
        sim = members[0][0]
        state["f"] = torch.zeros(sim.Q, sim.N, dtype=torch.float64, device="cuda")
    return state


class Batch:
    """The batch handle that a program keeps, given back with its state."""

    def __init__(self, lat, case, stream, sims):
        self.sims = sims  # outlive the handle
        self.handle = lbm.lbm_batch_create(lat, PRECISION[case["storage"]], case["order"], stream.cuda_stream, len(sims))
        lbm.lbm_batch_set_config(self.handle, 128, 1, case["graph_steps"])
        for sim in sims:
            lbm.lbm_batch_add(self.handle, sim.ctx)

    def __del__(self):
        lbm.lbm_batch_destroy(self.handle)


def run(state):
    case, use = state["case"], state["case"]["use"]
    out = dict(state["out"])
    if use == "batch":
        lbm.lbm_batch_step(state["batch"].handle, case["steps"])
        for sim, rho, u, T, q in state["sims"]:
            lbm.lbm_moments_async(sim.ctx, rho, u, T, q)
        return out
    sim, rho, u, T, q = state["sims"][0]
    if use in ("simulate", "monitor"):
        sim.init()
    if use == "monitor":
        sums = []
        for _ in range(case["steps"]):
            sim.step(1)
            _, mass, mom, energy = sim.conserved()
            sums.append([mass, *mom, energy])
        out["sums"] = np.array(sums)
    else:
        sim.step(case["steps"])
    lbm.lbm_moments_async(sim.ctx, rho, u, T, q)
    if use == "checkpoint":
        lbm.lbm_get_state(sim.ctx, state["f"])
        out["f"] = state["f"]
    return out


def work(case):
    """Every step reads and writes each population once (the next step needs all of them); fields are read where a pass
    begins with them, and written at its end. Operations of a site and step: 4 per direction for the moments, 12 for
    equilibrium, force and relaxation, and 60 for the site's own coefficients."""
    D = dims(case)
    Q = 37 if D == 2 else 39
    sites = sum(nx * ny * nz for nx, ny, nz, _, _ in grids(case, 0))
    if case["flow"] == "cylinders":
        sites *= 0.75  # the annulus
    step = 2 * Q * BYTES[case["storage"]] + (8 * D if FLOWS[case["flow"]][1] == "field" else 0)
    once = 8 * (2 + 2 * D) + Q * BYTES[case["storage"]]
    if case["use"] in ("simulate", "monitor"):
        once += 8 * (2 + D) + Q * BYTES[case["storage"]]
    if case["use"] == "checkpoint":
        once += 8 * Q + Q * BYTES[case["storage"]]
    per_step = step + (Q * BYTES[case["storage"]] if case["use"] == "monitor" else 0)
    return {"bytes": sites * (per_step * case["steps"] + once), "flops": sites * ((16 * Q + 60) * case["steps"] + 10 * Q)}


# ------------------------------------------------------------------ the same in 64 bits, with torch alone
# Velocity sets: one vector of each opposite pair (the rest particle first), in the order in which the populations are
# laid out in memory; shells (|e|^2 : weight) and the lattice constant.
D2Q37 = dict(D=2, neq=4, c=1.1969797703930743589723885, pairs=(
    (1, 0), (0, 1), (1, 1), (1, -1), (2, 0), (0, 2), (2, 1), (2, -1), (1, 2), (1, -2), (2, 2), (2, -2), (3, 0), (0, 3),
    (3, 1), (3, -1), (1, 3), (1, -3)), weights={
        0: 0.2331506691323525022865067, 1: 0.1073060915422190024124643, 2: 0.0576678598887948820300692,
        4: 0.0142082161584507502646989, 5: 0.0053530490005137752327315, 8: 0.0010119375926735754754109,
        9: 0.0002453010277577173454659, 10: 0.0002834142529941982174005})
D3Q39 = dict(D=3, neq=3, c=math.sqrt(1.5), pairs=(
    (1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 1), (1, 1, -1), (1, -1, 1), (1, -1, -1), (2, 0, 0), (0, 2, 0), (0, 0, 2),
    (2, 2, 0), (2, 0, 2), (2, 0, -2), (2, -2, 0), (0, 2, 2), (0, 2, -2), (3, 0, 0), (0, 3, 0), (0, 0, 3)), weights={
        0: 1 / 12, 1: 1 / 12, 3: 1 / 27, 4: 2 / 135, 8: 1 / 432, 9: 1 / 1620})


def velocities(lat):
    e = [(0,) * lat["D"]]
    for v in lat["pairs"]:
        e += [v, tuple(-a for a in v)]
    return e


class Exact:
    """Pull, collide with the Hermite equilibrium and force, half-way walls: f - w in double, [Q, nz, ny, nx]."""

    def __init__(self, case, p):
        self.lat = D2Q37 if p["D"] == 2 else D3Q39
        self.D, self.p, self.order = p["D"], p, case["order"]
        nx, ny, nz = p["shape"]
        self.dims = (nz, ny, nx)
        self.e = velocities(self.lat)
        self.Q = len(self.e)
        self.opp = [0] + [i + 1 if i % 2 else i - 1 for i in range(1, self.Q)]
        dev = p["rho"].device
        self.E = torch.tensor(self.e, dtype=torch.float64, device=dev)
        e2 = [sum(a * a for a in v) for v in self.e]
        self.w = torch.tensor([self.lat["weights"][k] for k in e2], dtype=torch.float64, device=dev).view(-1, 1)
        self.X2 = torch.tensor([float(k) for k in e2], dtype=torch.float64, device=dev).view(-1, 1) * self.lat["c"] ** 2
        self.n_wall = ny if self.D == 2 else nz
        self.dim_wall = 1 if self.D == 2 else 0  # of [nz, ny, nx]
        g = p["g"]
        N = p["N"]
        if g["kind"] == lbm.LBM_G_FIELD:
            self.g = g["field"]
        else:
            self.g = torch.tensor(g["g0"][:self.D], dtype=torch.float64, device=dev).view(self.D, 1)
            if g["kind"] == lbm.LBM_G_SINE:
                k = torch.arange(ny, dtype=torch.float64, device=dev).view(1, ny, 1).expand(nz, ny, nx).reshape(1, N)
                self.g = self.g * torch.sin(2.0 * math.pi * k / ny)
        self.solid = None if p["solid"] is None else torch.from_numpy(p["solid"].astype(bool)).to(dev)
        if self.solid is not None:
            self.Tw = torch.from_numpy(p["T_wall"]).to(dev)
        self.chunk = 1 << 21

    def over(self, N):
        return [slice(a, min(N, a + self.chunk)) for a in range(0, N, self.chunk)]

    def poly(self, rho, u, Th, g, tu):
        """(f0 / w - rho, F / w) at one set of sites; tu: xi . u for every direction."""
        D, X2 = self.D, self.X2
        u2, s, gu = (u * u).sum(0), self.lat["c"] * (self.E @ g), (g * u).sum(0)
        t2 = tu * tu
        Z = Th * (X2 - (D + 2)) - u2
        h = tu + 0.5 * (t2 - u2 + Th * (X2 - D)) + tu * (t2 + 3.0 * Z) / 6.0
        if self.lat["neq"] == 4:
            h += (t2 * t2 + 6.0 * t2 * (Th * (X2 - (D + 4)) - u2) + 3.0 * u2 * u2 - 6.0 * Th * u2 * (X2 - (D + 2))
                  + 3.0 * Th * Th * (X2 * X2 - 2.0 * (D + 2) * X2 + D * (D + 2))) / 24.0
        F = s
        if self.order >= 1:
            F = s * (1.0 + tu) - gu
        if self.order >= 2:
            F = s * (1.0 + tu + 0.5 * (t2 + Z)) - gu * (1.0 + tu)
        return rho * h, rho * F

    def g_of(self, sl):
        return self.g[:, sl] if self.g.shape[1] > 1 else self.g

    def state(self, d, g):
        """rho, u, theta - 1 at the middle of the step, and 1 / tau."""
        c, D = self.lat["c"], self.D
        m0 = d.sum(0)
        rho = 1.0 + m0
        ut = c * (self.E.T @ d) / rho
        k2 = (self.X2 * d).sum(0)
        Th = ((k2 - D * m0) / rho - (ut * ut).sum(0)) / D + (g * g).sum(0) / (4.0 * D)
        om = 1.0 / (self.p["mu"] / (rho * (1.0 + Th)) + 0.5) if self.p["mu"] > 0 else 1.0 / self.p["tau"]
        return m0, rho, ut + 0.5 * g, Th, om

    def start(self):
        """The populations whose first pull gives f~ = f0 - F / 2."""
        p, N = self.p, self.p["N"]
        f = torch.empty(self.Q, N, dtype=torch.float64, device=p["rho"].device)
        for sl in self.over(N):
            rho, u, g = p["rho"][sl], p["u"][:, sl], self.g_of(sl)
            h, F = self.poly(rho, u, p["T"][sl] - 1.0, g, self.lat["c"] * (self.E @ u))
            f[:, sl] = self.w * (rho - 1.0 + h - 0.5 * F)
        out = torch.zeros_like(f)
        n, dim = self.n_wall, self.dim_wall
        for i, e in enumerate(self.e):
            fi = f[i].view(self.dims)
            if self.p["wall"] == "periodic" or e[-1] == 0:
                back = tuple(-a for a in e)
                out[i] = self.source(f[i], back)
                if self.solid is not None:  # what the wall absorbs stays with the site
                    out[i] = torch.where(self.source(self.solid, back), f[i], out[i])
                continue
            a = e[-1]
            side = tuple(-b for b in reversed(e[:-1]))
            moved = torch.roll(fi, side, tuple(range(dim + 1, 3))) if side else fi
            o = out[i].view(self.dims)
            oo = out[self.opp[i]].view(self.dims)
            if a > 0:
                o.narrow(dim, 0, n - a).copy_(moved.narrow(dim, a, n - a))
                for r in range(a):
                    oo.select(dim, a - 1 - r).copy_(fi.select(dim, r))
            else:
                o.narrow(dim, -a, n + a).copy_(moved.narrow(dim, 0, n + a))
                for r in range(n + a, n):
                    oo.select(dim, 2 * n - 1 - (r - a)).copy_(fi.select(dim, r))
        return out

    def source(self, v, e):
        """v at x - e."""
        return torch.roll(v.view(self.dims), tuple(reversed(e)), tuple(range(3 - self.D, 3))).reshape(-1)

    def wall_f0(self, T):
        """f0(1, 0, T) / w - 1."""
        D, Th = self.D, T - 1.0
        h = 0.5 * Th * (self.X2 - D)
        if self.lat["neq"] == 4:
            h = h + Th * Th * (self.X2 * self.X2 - 2.0 * (D + 2) * self.X2 + D * (D + 2)) / 8.0
        return h

    def pull(self, f):
        out = torch.empty_like(f)
        n, dim = self.n_wall, self.dim_wall
        for i, e in enumerate(self.e):
            out[i] = self.source(f[i], e)
        if self.solid is not None:
            num, den, a0 = torch.zeros_like(out[0]), torch.zeros_like(out[0]), {}
            for i, e in enumerate(self.e):
                if not any(e):
                    continue
                hit = self.source(self.solid, e) & ~self.solid
                w, h = self.w[i, 0], self.wall_f0_at(i, self.source(self.Tw, e))
                num += torch.where(hit, f[self.opp[i]] - w * h, 0.0)
                den += torch.where(hit, w * (1.0 + h), 0.0)
                a0[i] = (hit, w, h)
            r = num / torch.where(den > 0, den, 1.0)
            for i, (hit, w, h) in a0.items():
                out[i] = torch.where(hit, w * (r * (1.0 + h) + h), out[i])
            return out
        if self.p["wall"] == "periodic":
            return out
        rho_w = {}
        if self.p["wall"] == "thermal":
            for low, T in ((True, self.p["T_lo"]), (False, self.p["T_hi"])):
                h = self.wall_f0(torch.tensor(T, dtype=torch.float64, device=f.device))
                got, w_in, h_in = 0.0, 0.0, 0.0
                for i, e in enumerate(self.e):
                    a = -e[-1] if low else e[-1]  # layers from which it leaves
                    for r in range(max(0, a)):
                        got = got + f[i].view(self.dims).select(dim, r if low else n - 1 - r)
                    for r in range(max(0, -a)):
                        w_in = w_in + self.w[i, 0] * (1.0 + h[i, 0])
                        h_in = h_in + self.w[i, 0] * h[i, 0]
                rho_w[low] = ((got - h_in) / w_in, h)
        for i, e in enumerate(self.e):
            a = e[-1]
            o, back = out[i].view(self.dims), f[self.opp[i]].view(self.dims)
            for r in (range(a) if a > 0 else range(n + a, n)):
                if self.p["wall"] == "bounce":
                    o.select(dim, r).copy_(back.select(dim, a - 1 - r if a > 0 else 2 * n - 1 - (r - a)))
                else:
                    m1, h = rho_w[a > 0]
                    o.select(dim, r).copy_(self.w[i, 0] * (m1 * (1.0 + h[i, 0]) + h[i, 0]))
        return out

    def wall_f0_at(self, i, T):
        D, Th, X2 = self.D, T - 1.0, self.X2[i, 0]
        h = 0.5 * Th * (X2 - D)
        if self.lat["neq"] == 4:
            h = h + Th * Th * (X2 * X2 - 2.0 * (D + 2) * X2 + D * (D + 2)) / 8.0
        return h

    def collide(self, d):
        """In place."""
        for sl in self.over(self.p["N"]):
            x, g = d[:, sl], self.g_of(sl)
            m0, rho, u, Th, om = self.state(x, g)
            h, F = self.poly(rho, u, Th, g, self.lat["c"] * (self.E @ u))
            d[:, sl] = x - om * (x - self.w * (m0 + h)) + (1.0 - 0.5 * om) * self.w * F
        if self.solid is not None:
            d[:, self.solid] = 0.0
        return d

    def fields(self, d):
        N = self.p["N"]
        new = lambda k: torch.empty(k, N, dtype=torch.float64, device=d.device)  # noqa: E731
        rho, u, T, q = new(1), new(self.D), new(1), new(self.D)
        c = self.lat["c"]
        for sl in self.over(N):
            x, g = d[:, sl], self.g_of(sl)
            m0, r, uu, Th, om = self.state(x, g)
            h, F = self.poly(r, uu, Th, g, c * (self.E @ uu))
            neq = x - self.w * (m0 + h) + 0.5 * self.w * F
            cc = c * self.E.unsqueeze(2) - uu.unsqueeze(0)  # Q, D, sites
            flux = (neq * (cc * cc).sum(1)).unsqueeze(1) * cc
            rho[0, sl], u[:, sl], T[0, sl] = r, uu, 1.0 + Th
            q[:, sl] = 0.5 * (1.0 - 0.5 * om) * flux.sum(0)
        if self.solid is not None:
            for v in (rho, u, T, q):
                v[:, self.solid] = 0.0
        return {"rho": rho.reshape(-1), "u": u.reshape(-1), "T": T.reshape(-1), "q": q.reshape(-1)}

    def sums(self, d):
        r = self.fields(d)
        u = r["u"].view(self.D, -1)
        mom = [float((r["rho"] * v).sum()) for v in u]
        return [float(r["rho"].sum()), *mom, float((r["rho"] * ((u * u).sum(0) + self.D * r["T"])).sum() * 0.5)]


def exact(case, seed):
    parts, sums, f = [], [], None
    for k, grid in enumerate(grids(case, seed)):
        x = Exact(case, problem(case, grid, seed * 1009 + k))
        f = x.start()
        for _ in range(case["steps"]):
            f = x.collide(x.pull(f))
            if case["use"] == "monitor":
                sums.append(x.sums(x.pull(f)))
        parts.append(x.fields(x.pull(f)))
    out = {k: torch.cat([p[k] for p in parts]) for k in ("rho", "u", "T", "q")}
    if case["use"] == "monitor":
        out["sums"] = np.array(sums)
    if case["use"] == "checkpoint":
        out["f"] = f + x.w
    return out
