"""Workloads of the viscous solver, as a program that uses it runs them.

Each case is one call sequence of a simulation through ``paper_2206_14780_gb300.binding`` on
synthetic particles drawn from a seed:

* ``step``   one full predictor/corrector time step (``Stepper.step``);
* ``solve``  one implicit solve of a time-step loop: neighbour rebuild at the new positions, the
             viscosity pass or the learned row scale where the case has one, the start from the
             previous velocity, the solve, and the float32 velocities the program keeps;
* ``host``   the same from host buffers (``solve_host``);
* ``apply``  one operator application on a set-up operator, as an outer solver calls it;
* ``batch``  an ensemble of scenes solved together (``Batch.solve``);
* ``train``  loss and gradient of the network over a set of particles (``Mlp.grad``).

Geometries are the channel, the open box and the inclined slope, on lattices of any extent, with
the Wendland kernel (about 80 neighbours) or the truncated Gaussian (about 250).  Solves stop at a
1e-8 true residual, as the flow simulations do: the velocities are then good to float32.
"""
import math
import os

import numpy as np
import torch

import paper_2206_14780_gb300 as package
from paper_2206_14780_gb300 import binding

DX = 0.005
RHO0 = 1000.0
GAUSS_K = 3.0
GAUSS_W = math.pi ** 1.5 * math.erf(GAUSS_K) - 2.0 * math.pi / 3.0 * math.exp(-GAUSS_K ** 2) * GAUSS_K * (
    3.0 + 2.0 * GAUSS_K ** 2)
RTOL = 1e-8


# ---- the cases --------------------------------------------------------------------------------

def listed():
    return [
        # the narrow plane channel of the flow tables at 16 spacings across: the smallest system a
        # user steps (thousands of steps per run), dummy walls, Newtonian
        dict(name="step_channel_1k", kind="step", shape="channel", nx=8, ny=16, nz=8, kernel="wendland",
             boundary="dummy", bingham=False),
        # a regularised Bingham fluid between dynamic walls, Gaussian kernel, 32 across
        dict(name="step_bingham_6k", kind="step", shape="channel", nx=12, ny=31, nz=12, kernel="gaussian",
             boundary="dynamic", bingham=True),
        # a larger time step: jittered channel with ragged extents, caller order mixed by motion
        dict(name="step_channel_91k", kind="step", shape="channel", nx=45, ny=37, nz=47, kernel="wendland",
             boundary="dummy", bingham=False),
        # the small Couette channel from pinned host buffers, the call of a host-side integrator
        dict(name="host_couette_3k", kind="host", shape="channel", nx=20, ny=10, nz=10, kernel="wendland",
             boundary="dummy", nu=1.0, dt=1e-4),
        # slope flow with shear-dependent viscosity: the mu pass, then a stiff solve
        dict(name="solve_slope_58k", kind="solve", shape="slope", nx=50, ny=20, nz=50, kernel="wendland",
             boundary="dummy", mean="harmonic", rheology=True, dt=5e-4, shuffled=False),
        # lava-like box at a ragged mid size, particles in mixed order, arithmetic mean viscosity,
        # preconditioned with the learned wall-row scale
        dict(name="solve_box_95k", kind="solve", shape="box", nx=41, ny=38, nz=43, kernel="wendland",
             boundary="dummy", mean="arithmetic", nu=10.0, dt=5e-4, shuffled=True, scale="learned"),
        # the same kind of box with the truncated Gaussian kernel: rows of ~250 neighbours
        dict(name="solve_gauss_77k", kind="solve", shape="box", nx=36, ny=36, nz=36, kernel="gaussian",
             boundary="dummy", mean="harmonic", nu=10.0, dt=5e-4, shuffled=False),
        # conjugate gradient on the symmetric system of a wide channel between dynamic walls
        dict(name="solve_cg_channel_416k", kind="solve", shape="channel", nx=119, ny=30, nz=97, kernel="wendland",
             boundary="dynamic", mean="harmonic", nu=100.0, dt=5e-4, method="cg", shuffled=False),
        # the large box, 100^3 fluid particles on a floor between walls: the benchmark's solve
        dict(name="solve_box_1157k", kind="solve", shape="box", nx=100, ny=100, nz=100, kernel="wendland",
             boundary="dummy", mean="harmonic", nu=10.0, dt=5e-4, shuffled=False),
        # the operator alone at a size with a ragged last slice
        dict(name="apply_box_274k", kind="apply", shape="box", nx=61, ny=59, nz=60, kernel="wendland",
             boundary="dummy", mean="harmonic", nu=10.0, dt=5e-4, shuffled=True),
        # an ensemble of unequal scenes in one batched solve
        dict(name="batch_16_scenes", kind="batch", scenes=16, lo=10000, hi=120000, kernel="wendland"),
        # the scale network's training gradient over the particles of a scene
        dict(name="train_262k", kind="train", rows=262147),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _extents(rng, total, least):
    """Three lattice extents of about `total` particles, none below `least`, of uneven ratios."""
    side = total ** (1.0 / 3.0)
    a, c = (math.exp(rng.uniform(-0.35, 0.35)) for _ in range(2))
    e = [side * a, side / (a * c), side * c]
    return [max(least, int(round(v))) for v in e]


def draw(rng):
    kind = rng.choice(["step", "step", "solve", "solve", "solve", "solve", "host", "apply", "batch", "train"])
    if kind == "train":
        return dict(kind="train", rows=_log_int(rng, 2000, 1000000))
    if kind == "batch":
        return dict(kind="batch", scenes=rng.randint(3, 24), lo=_log_int(rng, 4000, 20000),
                    hi=_log_int(rng, 30000, 120000), kernel="wendland")
    gauss = rng.random() < 0.25
    least = 12 if gauss else 8
    kernel = "gaussian" if gauss else "wendland"
    if kind == "step":
        nx, ny, nz = _extents(rng, _log_int(rng, 1000, 40000 if gauss else 120000), least)
        return dict(kind="step", shape="channel", nx=nx, ny=ny, nz=nz, kernel=kernel,
                    boundary=rng.choice(["dummy", "dynamic"]), bingham=rng.random() < 0.4)
    shape = rng.choice(["channel", "box", "slope"] if kind == "solve" else ["channel", "box"])
    most = {"host": 100000, "apply": 900000, "solve": 200000 if shape == "slope" else 700000}[kind] // (4 if gauss else 1)
    nx, ny, nz = _extents(rng, _log_int(rng, 1200, most), least)
    case = dict(kind=kind, nx=nx, ny=ny, nz=nz, kernel=kernel, dt=math.exp(rng.uniform(math.log(1e-4), math.log(5e-4))),
                nu=math.exp(rng.uniform(math.log(1.0), math.log(30.0))), mean=rng.choice(["harmonic", "arithmetic"]),
                shuffled=rng.random() < 0.5)
    case["shape"] = shape
    case["boundary"] = rng.choice(["dummy", "dummy", "dynamic"])
    if kind == "host":   # solve_host takes the Wendland kernel
        case["kernel"] = "wendland"
    if case["shape"] == "slope":
        case["rheology"] = True
        case["nu"] = 1.0
    if kind == "solve":
        if case["boundary"] == "dynamic" and rng.random() < 0.5:
            case["method"] = "cg"
        elif case["boundary"] == "dummy" and rng.random() < 0.3:
            case["scale"] = "learned"
        elif rng.random() < 0.15 and nx * ny * nz < 60000:
            case["precision"] = "fp64"
    return case


# ---- particles --------------------------------------------------------------------------------

def _lattice(nx, ny, nz, origin=(0.0, 0.0, 0.0)):
    """Positions ((i, j, k) + 1/2 + origin) in spacings, float64 on the GPU."""
    ax = [torch.arange(k, dtype=torch.float64, device="cuda") + 0.5 + o for k, o in zip((nx, ny, nz), origin)]
    return torch.stack(torch.meshgrid(*ax, indexing="ij"), dim=-1).reshape(-1, 3)


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _geometry(case):
    """Fluid and wall positions in spacings, the box and its periodic axes."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    layers = 4 if case["kernel"] == "gaussian" else 3
    fluid = _lattice(nx, ny, nz)
    if case["shape"] == "channel":      # walls normal to y, periodic in x and z
        walls = [_lattice(nx, layers, nz, (0, -layers, 0)), _lattice(nx, layers, nz, (0, ny, 0))]
        return fluid, torch.cat(walls), (0, -layers, 0), (nx, ny + layers, nz), (1, 0, 1)
    if case["shape"] == "slope":        # a floor normal to y, free surface, periodic in x and z
        return fluid, _lattice(nx, layers, nz, (0, -layers, 0)), (0, -layers, 0), (nx, ny + 4, nz), (1, 0, 1)
    mx, my = nx + 2 * layers, ny + 2 * layers   # floor and four side walls, open top (z)
    walls = [_lattice(mx, my, layers, (-layers, -layers, -layers)), _lattice(layers, my, nz, (-layers, -layers, 0)),
             _lattice(layers, my, nz, (nx, -layers, 0)), _lattice(nx, layers, nz, (0, -layers, 0)),
             _lattice(nx, layers, nz, (0, ny, 0))]
    return (fluid, torch.cat(walls), (-layers, -layers, -layers), (nx + layers, ny + layers, nz + 4), (0, 0, 0))


def _scene(case, seed):
    """A solve's particles: positions with mass, density, viscosity, types, velocities, right-hand side."""
    g = _generator(seed)
    fluid, walls, lo, hi, periodic = _geometry(case)
    nf, n = fluid.shape[0], fluid.shape[0] + walls.shape[0]
    ny = case["ny"]
    # the particles have moved off the lattice: +-0.1 spacings
    fluid = fluid + (torch.rand(fluid.shape, generator=g, dtype=torch.float64, device="cuda") - 0.5) * 0.2
    noise = torch.randn(fluid.shape, generator=g, dtype=torch.float64, device="cuda")
    v, wall_v, grav = torch.zeros_like(fluid), torch.zeros_like(walls), torch.zeros(3, dtype=torch.float64, device="cuda")
    mu = torch.full((n,), RHO0 * case.get("nu", 1.0), dtype=torch.float32, device="cuda")
    if case["shape"] == "channel":
        v[:, 0] = fluid[:, 1] / ny
        v += 0.01 * noise
        wall_v[walls[:, 1] > 0, 0] = 1.0
    elif case["shape"] == "slope":       # sheared layer under a rigid plug, gravity turned by 10 degrees
        y0 = 2.0 * ny / 3.0
        v[:, 0] = 0.1 * (1.0 - (1.0 - fluid[:, 1].clamp(0.0, y0) / y0) ** 2) * (1.0 + 1e-5 * noise[:, 0])
        v[:, 1:] = 1e-6 * noise[:, 1:]
        th = math.radians(10.0)
        grav = torch.tensor([9.81 * math.sin(th), -9.81 * math.cos(th), 0.0], dtype=torch.float64, device="cuda")
    else:
        v = 0.1 * noise
    pos = torch.zeros((n, 4), dtype=torch.float32, device="cuda")
    pos[:, :3] = _fold(torch.cat([fluid, walls]) * DX, lo, hi, periodic, DX)
    pos[:, 3] = RHO0 * DX ** 3
    ptype = torch.zeros(n, dtype=torch.uint8, device="cuda")
    ptype[nf:] = 1
    vel = torch.zeros((n, 4), dtype=torch.float32, device="cuda")
    vel[:, :3] = torch.cat([v, wall_v])
    if case.get("shuffled"):
        p = torch.randperm(n, generator=g, device="cuda")
        pos, ptype, vel, mu = pos[p].contiguous(), ptype[p].contiguous(), vel[p].contiguous(), mu[p].contiguous()
    wall = (ptype != 0)[:, None]
    v64 = vel[:, :3].double()
    b = torch.where(wall, (2.0 if case["boundary"] == "dummy" else 1.0) * v64, v64 + case["dt"] * grav)
    return dict(pos=pos, rho=torch.full((n,), RHO0, dtype=torch.float32, device="cuda"), mu=mu, ptype=ptype, vel=vel,
                b=b.contiguous(), lo=[x * DX for x in lo], hi=[x * DX for x in hi], periodic=list(periodic),
                h=float(np.float32(1.3 * DX)), kernel=1 if case["kernel"] == "gaussian" else 0)


def _fold(p, lo, hi, periodic, dx):
    """float32 positions inside [lo, hi) on the periodic axes."""
    p = p.clone()
    for ax in range(3):
        if periodic[ax]:
            a, length = lo[ax] * dx, (hi[ax] - lo[ax]) * dx
            p[:, ax] = a + torch.remainder(p[:, ax] - a, length)
    p = p.float()
    for ax in range(3):
        if periodic[ax]:
            p[:, ax] = torch.where(p[:, ax] >= np.float32(hi[ax] * dx), float(np.float32(lo[ax] * dx)), p[:, ax])
    return p


def _flow(case, seed):
    """A time step's state: a channel driven by a body force, near its developed profile."""
    g = _generator(seed)
    fluid, walls, lo, hi, periodic = _geometry(case)
    nf, n, ny = fluid.shape[0], fluid.shape[0] + walls.shape[0], case["ny"]
    dp, mu0, force = 1.0 / ny, 0.1, 0.05
    fluid = fluid + (torch.rand(fluid.shape, generator=g, dtype=torch.float64, device="cuda") - 0.5) * 0.02
    y = fluid[:, 1] * dp
    v = torch.zeros_like(fluid)
    v[:, 0] = force / (2 * mu0) * y * (1.0 - y)
    v += 1e-4 * torch.randn(fluid.shape, generator=g, dtype=torch.float64, device="cuda")
    flat = torch.zeros(10 * n, dtype=torch.float32, device="cuda")   # pos, vel, rho, mu
    flat[:4 * n].view(n, 4)[:, :3] = _fold(torch.cat([fluid, walls]) * dp, lo, hi, periodic, dp)
    flat[:4 * n].view(n, 4)[:, 3] = dp ** 3
    flat[4 * n:8 * n].view(n, 4)[:nf, :3] = v.float()
    flat[8 * n:9 * n] = 1.0 + 1e-5 * torch.randn(n, generator=g, device="cuda")
    flat[9 * n:] = mu0
    ptype = torch.zeros(n, dtype=torch.uint8, device="cuda")
    ptype[nf:] = 1
    h, c0 = float(np.float32(1.3 * dp)), 6.32
    return dict(flat=flat, ptype=ptype, n=n, lo=[x * dp for x in lo], hi=[x * dp for x in hi], periodic=list(periodic),
                h=h, kernel=1 if case["kernel"] == "gaussian" else 0, dt=0.3 * h / c0, rho0=1.0, c0=c0, zeta=7.0,
                g=(force, 0.0, 0.0), rheology=(0.0125, mu0, 1000.0) if case["bingham"] else None)


def _capacity(case):
    return 320 if case["kernel"] == "gaussian" else 128


def _params(case):
    return binding.visc_params(case["dt"], binding.SPH_BC_DUMMY if case["boundary"] == "dummy" else binding.SPH_BC_DYNAMIC,
                               binding.SPH_MEAN_ARITHMETIC if case.get("mean") == "arithmetic" else binding.SPH_MEAN_HARMONIC)


def _opts(case):
    return binding.solve_opts(rtol=RTOL, method=1 if case.get("method") == "cg" else 0,
                              precision=binding.SPH_PREC_FP64 if case.get("precision") == "fp64" else binding.SPH_PREC_MIXED)


BINGHAM = (100.0, 1e3, 1000.0)   # the slope's yield stress, plastic viscosity and regularisation


def _members(case):
    """The scenes of an ensemble: channels and boxes of log-spaced sizes, viscosities and time steps."""
    out = []
    for k in range(case["scenes"]):
        f = k / max(1, case["scenes"] - 1)
        total = case["lo"] * (case["hi"] / case["lo"]) ** f
        side = max(8, int(round((0.7 * total) ** (1.0 / 3.0))))
        nu, dt = math.exp(math.log(300.0) * ((k * 5) % 11) / 10.0), 1e-4 * 5.0 ** (((k * 3) % 7) / 6.0)
        shape = dict(shape="channel", nx=side + 3, ny=max(6, side - 5), nz=side + 2) if k % 2 == 0 else dict(
            shape="box", nx=side, ny=side + 1, nz=side - 1)
        out.append(dict(shape, kernel=case["kernel"], boundary="dummy", mean="harmonic", nu=nu, dt=dt))
    return out


def _network(seed):
    """Network parameters as at the start of training: weights of variance 1 / fan-in, small biases."""
    g = _generator(seed + 1)
    out = []
    for fan_in, fan_out in ((16, 64), (64, 64), (64, 64), (64, 3)):
        out.append(torch.randn(fan_out * fan_in, generator=g, device="cuda") / math.sqrt(fan_in))
        out.append(0.1 * torch.randn(fan_out, generator=g, device="cuda"))
    return torch.cat(out)


def _rows(case, seed):
    """Features, targets and mask of a training set."""
    g = _generator(seed)
    m = case["rows"]
    feats = torch.randn((m, 16), generator=g, device="cuda").bfloat16()
    targets = torch.randn((m, 4), generator=g, device="cuda")
    targets[:, 3] = 0.0
    mask = (torch.rand(m, generator=g, device="cuda") < 0.9).to(torch.uint8)
    return feats, targets, mask


# ---- what a program has in hand, and one pass -------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    if kind == "train":
        feats, targets, mask = _rows(case, seed)
        return dict(kind=kind, mlp=binding.Mlp(_network(seed).cpu().numpy()), feats=feats.view(torch.int16), targets=targets,
                    mask=mask, count=int(mask.sum()), grad=torch.empty(binding.MLP_NPARAMS, device="cuda"),
                    loss=torch.empty(1, device="cuda"))
    if kind == "step":
        f = _flow(case, seed)
        n, work = f["n"], f["flat"].clone()
        views = [work[:4 * n].view(n, 4), work[4 * n:8 * n].view(n, 4), work[8 * n:9 * n], work[9 * n:]]
        stepper = binding.Stepper(*views, f["ptype"], f["lo"], f["hi"], f["periodic"], f["h"], kernel=f["kernel"])
        params = binding.step_params(f["dt"], f["rho0"], f["c0"], f["zeta"], f["g"],
                                     binding.SPH_BC_DUMMY if case["boundary"] == "dummy" else binding.SPH_BC_DYNAMIC,
                                     rheology=f["rheology"], max_neighbors=_capacity(case))
        return dict(kind=kind, start=f["flat"], work=work, views=views, stepper=stepper, params=params, opts=_opts(case))
    if kind == "batch":
        members = []
        for k, c in enumerate(_members(case)):
            s = _scene(c, seed * 64 + k)
            s["params"] = _params(c)
            s["nb"] = binding.build_neighbors(*_particles(s), _capacity(c), kernel=s["kernel"])
            s["x"] = torch.empty_like(s["b"])
            members.append(s)
        batch = binding.Batch([s["nb"] for s in members], [s["params"] for s in members])
        return dict(kind=kind, members=members, batch=batch, opts=_opts(case))
    s = _scene(case, seed)
    s.update(kind=kind, params=_params(case), opts=_opts(case), capacity=_capacity(case))
    if kind == "host":
        for name in ("pos", "rho", "mu", "ptype", "vel", "b"):
            s[name] = s[name].cpu().pin_memory()
        s["x"] = torch.empty_like(s["b"], pin_memory=True)
        s["nb"] = None
        return s
    s["nb"] = binding.build_neighbors(*_particles(s), s["capacity"], kernel=s["kernel"])
    if kind == "apply":
        s["nb"].setup(s["params"])
        s["out"] = torch.empty_like(s["vel"])
        return s
    s["x"] = torch.empty_like(s["b"])
    s["out"] = torch.zeros_like(s["vel"])
    s["rheology"] = BINGHAM if case.get("rheology") else None
    s["mlp"] = None
    if case.get("scale") == "learned":
        with np.load(os.path.join(os.path.dirname(package.__file__), "weights", "scale_head_mlp.npz")) as w:
            s["mlp"] = binding.Mlp(w["params"])
    return s


def _particles(s):
    return s["pos"], s["rho"], s["mu"], s["ptype"], s["lo"], s["hi"], s["periodic"], s["h"]


def run(state):
    s, kind = state, state["kind"]
    if kind == "solve":
        nb = s["nb"]
        nb.rebuild(*_particles(s), s["capacity"], kernel=s["kernel"])
        if s["rheology"]:
            nb.mu_papanastasiou(s["vel"], s["vel"], *s["rheology"], s["mu"], set_handle=True)
        if s["mlp"] is not None:
            binding.mlp_row_scale(nb, s["params"], s["mlp"], s["vel"], None)
        binding.warm_start(nb, s["params"], None, s["vel"], s["ptype"], s["b"], s["x"])
        nb.solve(s["params"], s["opts"], s["b"], s["x"], raise_on_nonconvergence=True)
        s["out"][:, :3] = s["x"]
        return dict(vel=s["out"], mu=s["mu"]) if s["rheology"] else dict(vel=s["out"])
    if kind == "step":
        s["work"].copy_(s["start"])     # every pass steps from the same state
        s["stepper"].step(s["params"], s["opts"])
        return dict(zip(("pos", "vel", "rho", "mu"), s["views"]))
    if kind == "host":
        _, s["nb"] = binding.solve_host(*_particles(s), s["params"], s["opts"], s["vel"], s["b"], s["x"], nb=s["nb"],
                                        max_neighbors=s["capacity"])
        return dict(vel=s["x"].float())
    if kind == "apply":
        s["nb"].apply(s["params"], s["vel"], s["out"])
        return dict(out=s["out"])
    if kind == "batch":
        for m in s["members"]:
            m["x"].copy_(m["vel"][:, :3])
        s["batch"].solve(s["opts"], [m["b"] for m in s["members"]], [m["x"] for m in s["members"]])
        return [m["x"].float() for m in s["members"]]
    s["mlp"].grad(s["feats"], s["targets"], s["mask"], s["count"], s["grad"], s["loss"])
    return dict(grad=s["grad"], loss=s["loss"])


def _count(case):
    """(particles, of them fluid) of a geometry, without making it."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    layers = 4 if case["kernel"] == "gaussian" else 3
    fluid = nx * ny * nz
    if case["shape"] == "channel":
        return fluid + 2 * layers * nx * nz, fluid
    if case["shape"] == "slope":
        return fluid + layers * nx * nz, fluid
    mx, my = nx + 2 * layers, ny + 2 * layers
    return fluid + layers * mx * my + 2 * layers * my * nz + 2 * layers * nx * nz, fluid


def work(case):
    """Inputs and outputs once; per pair the coefficient (about 25 operations) and two applications of the operator
    (the first residual and the accepting one: 12 operations a pair each)."""
    kind = case["kind"]
    if kind == "train":
        return dict(bytes=case["rows"] * (32 + 16 + 1) + 4 * 9604, flops=case["rows"] * 56064)
    members = _members(case) if kind == "batch" else [case]
    total = dict(bytes=0, flops=0)
    for c in members:
        n, _ = _count(c)
        pairs = n * (220 if c["kernel"] == "gaussian" else 72)
        if kind == "apply":
            total["bytes"] += 8 * pairs + 32 * n
            total["flops"] += 12 * pairs
        elif kind == "step":
            total["bytes"] += 81 * n
            total["flops"] += 2 * 49 * pairs
        else:
            total["bytes"] += (16 + 4 + 4 + 1 + 16 + 24 + 24) * n
            total["flops"] += 49 * pairs
    return total


# ---- the same in 64 bits, in plain torch ------------------------------------------------------

def _pairs(pos, lo, hi, periodic, radius):
    """(i, j, r_j - r_i) of all pairs closer than radius, both directions, positions float64."""
    n, dev = pos.shape[0], pos.device
    cells, index = [], []
    for ax in range(3):
        length = hi[ax] - lo[ax]
        nc = max(1, int(math.floor(length / (radius * (1.0 + 1e-6)))))
        c = torch.floor((pos[:, ax] - lo[ax]) * (nc / length)).long()
        index.append(torch.remainder(c, nc) if periodic[ax] else c.clamp(0, nc - 1))
        cells.append(nc)
    key = index[0] + cells[0] * (index[1] + cells[1] * index[2])
    order = torch.argsort(key, stable=True)
    count = torch.bincount(key, minlength=cells[0] * cells[1] * cells[2])
    start = torch.cumsum(count, 0) - count
    found = []
    for dz in (-1, 0, 1):
        for dy in (-1, 0, 1):
            for dx in (-1, 0, 1):
                at, keep = [], torch.ones(n, dtype=torch.bool, device=dev)
                for ax, d in enumerate((dx, dy, dz)):
                    c = index[ax] + d
                    if periodic[ax]:
                        c = torch.remainder(c, cells[ax])
                    else:
                        keep &= (c >= 0) & (c < cells[ax])
                    at.append(c.clamp(0, cells[ax] - 1))
                cell = at[0] + cells[0] * (at[1] + cells[1] * at[2])
                many = torch.where(keep, count[cell], 0)
                i = torch.repeat_interleave(torch.arange(n, device=dev), many)
                first = torch.cumsum(many, 0) - many
                j = order[start[cell][i] + torch.arange(i.numel(), device=dev) - first[i]]
                d = pos[j] - pos[i]
                for ax in range(3):
                    if periodic[ax]:
                        length = hi[ax] - lo[ax]
                        d[:, ax] -= length * torch.round(d[:, ax] / length)
                near = ((d * d).sum(1) < radius * radius) & (i != j)
                found.append((i[near], j[near], d[near]))
    return tuple(torch.cat([f[k] for f in found]) for k in range(3))


class _System:
    """The viscous matrix A(dt) of a particle set in float64."""

    def __init__(self, pos, mass, rho, ptype, lo, hi, periodic, h, kernel):
        self.n, self.h, self.kernel = pos.shape[0], h, kernel
        self.mass, self.rho, self.fluid = mass, rho, ptype == 0
        self.i, self.j, self.d = _pairs(pos, lo, hi, periodic, (GAUSS_K if kernel else 2.0) * h)
        self.q = torch.sqrt((self.d * self.d).sum(1)) / h

    def grad_w(self):
        """|F| of every pair: the gradient of W is |F| (r_a - r_b)."""
        if self.kernel:
            return 2.0 / GAUSS_W * torch.exp(-self.q ** 2) / self.h ** 5
        return 105.0 / (128.0 * math.pi) * (2.0 - self.q).clamp(min=0) ** 3 / self.h ** 5

    def w(self):
        if self.kernel:
            return (torch.exp(-self.q ** 2) - math.exp(-GAUSS_K ** 2)) / GAUSS_W / self.h ** 3
        return 21.0 / (16.0 * math.pi) * (1.0 - 0.5 * self.q).clamp(min=0) ** 4 * (2.0 * self.q + 1.0) / self.h ** 3

    def sum(self, values):
        """Pair values added up over the row particle."""
        out = torch.zeros((self.n,) + values.shape[1:], dtype=torch.float64, device=values.device)
        return out.index_add_(0, self.i, values)

    def matrix(self, mu, dt, dummy, arithmetic):
        """A(dt) as CSR, and its Jacobi diagonal."""
        i, j = self.i, self.j
        fi, fj = self.fluid[i], self.fluid[j]
        mean = 0.5 * (mu[i] + mu[j]) if arithmetic else 2.0 * mu[i] * mu[j] / (mu[i] + mu[j])
        mean = torch.where(fj, mean, mu[i])
        a = torch.where(fi, 2.0 * dt * mean * self.mass[j] * self.grad_w() / (self.rho[i] * self.rho[j]), 0.0)
        diag = 1.0 + self.sum(a)
        values = -a
        if dummy:
            wall = ~fi & fj
            w = torch.where(wall, self.w(), 0.0)
            s = self.sum(w)
            values = torch.where(wall, w / torch.where(s > 0, s, 1.0)[i], values)
        every = torch.arange(self.n, device=i.device)
        keep = values != 0
        rows, cols = torch.cat([i[keep], every]), torch.cat([j[keep], every])
        values = torch.cat([values[keep], diag])
        order = torch.argsort(rows * self.n + cols)
        crow = torch.zeros(self.n + 1, dtype=torch.int64, device=i.device)
        crow[1:] = torch.cumsum(torch.bincount(rows, minlength=self.n), 0)
        return torch.sparse_csr_tensor(crow, cols[order], values[order], (self.n, self.n)), diag

    def viscosity(self, vel, tau0, mu0, m):
        """Papanastasiou viscosity of every fluid particle (mu0 on walls)."""
        f = (self.mass / self.rho)[self.j] * self.grad_w()
        du = vel[self.j] - vel[self.i]
        grad = torch.stack([self.sum((f * self.d[:, k])[:, None] * du) for k in range(3)], 1)
        sym = 0.5 * (grad + grad.transpose(1, 2))
        rate = torch.sqrt(2.0 * (sym * sym).sum((1, 2)))
        x = m * rate
        y = torch.where(x > 0, -torch.expm1(-x) / rate.clamp(min=1e-300), m)
        return torch.where(self.fluid, tau0 * y + mu0, mu0)


def _bicgstab(a, diag, b, x):
    """x of A x = b to the end of float64: restarted BiCGSTAB on the Jacobi-scaled system, three columns at once."""
    norm = torch.linalg.norm(b)
    best, best_x = float("inf"), x
    for _ in range(12):
        true = b - a @ x
        now = float(torch.linalg.norm(true) / norm) if float(norm) else 0.0
        if now < best:
            better, best, best_x = now < 0.3 * best, now, x
            if not better:
                break
        else:
            break
        if best < 1e-14:
            break
        r = true / diag[:, None]
        r0, p, rho = r.clone(), r.clone(), (r * r).sum(0)
        goal = 1e-7 * torch.linalg.norm(r)
        for k in range(3000):
            ap = (a @ p) / diag[:, None]
            alpha = rho / (r0 * ap).sum(0)
            alpha = torch.where(torch.isfinite(alpha), alpha, 0.0)
            s = r - alpha * ap
            t = (a @ s) / diag[:, None]
            omega = (t * s).sum(0) / (t * t).sum(0)
            omega = torch.where(torch.isfinite(omega), omega, 0.0)
            x = x + alpha * p + omega * s
            r = s - omega * t
            if k % 8 == 7 and float(torch.linalg.norm(r)) <= float(goal):
                break
            new = (r0 * r).sum(0)
            beta = new / rho * alpha / omega
            beta = torch.where(torch.isfinite(beta), beta, 0.0)
            p = r + beta * (p - omega * ap)
            rho = new
    return best_x


def _solution(case, s):
    system = _System(s["pos"][:, :3].double(), s["pos"][:, 3].double(), s["rho"].double(), s["ptype"], s["lo"], s["hi"],
                     s["periodic"], s["h"], s["kernel"])
    mu = s["mu"].double()
    if case.get("rheology"):
        mu = system.viscosity(s["vel"][:, :3].double(), *BINGHAM)
    a, diag = system.matrix(mu, case["dt"], case["boundary"] == "dummy", case.get("mean") == "arithmetic")
    return a, diag, mu


def _exact_step(case, seed):
    f = _flow(case, seed)
    n, flat, dt, dummy = f["n"], f["flat"].double(), f["dt"], case["boundary"] == "dummy"
    pos, mass, vel = flat[:4 * n].view(n, 4)[:, :3], flat[:4 * n].view(n, 4)[:, 3], flat[4 * n:8 * n].view(n, 4)[:, :3]
    rho, mu, fluid = flat[8 * n:9 * n], flat[9 * n:], (f["ptype"] == 0)
    g = torch.tensor(f["g"], dtype=torch.float64, device="cuda")
    scale = f["c0"] ** 2 * f["rho0"] / f["zeta"]

    def fold(p):
        for ax in range(3):
            if f["periodic"][ax]:
                length = f["hi"][ax] - f["lo"][ax]
                p[:, ax] = f["lo"][ax] + torch.remainder(p[:, ax] - f["lo"][ax], length)
        return p

    def forces(at, u, density, viscosity, scaled_dt):
        """Acceleration, density rate and densities (dummy walls from the closure), viscosity, next velocities."""
        system = _System(at, mass, density, f["ptype"], f["lo"], f["hi"], f["periodic"], f["h"], f["kernel"])
        if f["rheology"]:
            viscosity = system.viscosity(u, *f["rheology"])
        i, j, d = system.i, system.j, system.d
        pressure = scale * ((density / f["rho0"]) ** f["zeta"] - 1.0)
        if dummy:
            w = torch.where(~fluid[i] & fluid[j], system.w(), 0.0)
            total = system.sum(w)
            num = system.sum(w * (pressure[j] - (d @ g) * density[j]))
            wall_p = torch.where(total > 0, num / torch.where(total > 0, total, 1.0), 0.0)
            pressure = torch.where(fluid, pressure, wall_p)
            density = torch.where(fluid, density, f["rho0"] * (wall_p / scale + 1.0) ** (1.0 / f["zeta"]))
            system.rho = density
        mf = system.mass[j] * system.grad_w()
        term = pressure / density ** 2
        acc = torch.where(fluid[:, None], g - system.sum((mf * (term[i] + term[j]))[:, None] * d), 0.0)
        rate = system.sum(mf * ((u[i] - u[j]) * d).sum(1))
        if dummy:
            rate = torch.where(fluid, rate, 0.0)
        a, diag = system.matrix(viscosity, scaled_dt, dummy, False)
        b = torch.where(fluid[:, None], vel + scaled_dt * acc, (2.0 if dummy else 1.0) * vel)
        x = _bicgstab(a, diag, b, u.clone())
        return rate, density, viscosity, torch.where(fluid[:, None], x, vel)

    rate, rho0, mu, half = forces(pos, vel, rho, mu, 0.5 * dt)
    at = fold(pos + 0.5 * dt * vel)
    rate, _, mu, new = forces(at, half, rho0 + 0.5 * dt * rate, mu, dt)
    four = torch.zeros((n, 4), dtype=torch.float64, device="cuda")
    moved, speed = four.clone(), four
    moved[:, :3], moved[:, 3] = fold(pos + 0.5 * dt * (vel + new)), mass
    speed[:, :3] = new
    return dict(pos=moved, vel=speed, rho=rho0 + dt * rate, mu=mu)


def exact(case, seed):
    kind = case["kind"]
    if kind == "step":
        return _exact_step(case, seed)
    if kind == "batch":
        out = []
        for k, c in enumerate(_members(case)):
            s = _scene(c, seed * 64 + k)
            a, diag, _ = _solution(c, s)
            out.append(_bicgstab(a, diag, s["b"], s["vel"][:, :3].double()))
        return out
    if kind == "train":
        feats, targets, mask = _rows(case, seed)
        p = _network(seed).double().requires_grad_(True)
        x, at = feats.double(), 0
        for fan_in, fan_out in ((16, 64), (64, 64), (64, 64), (64, 3)):
            w, at = p[at:at + fan_out * fan_in].view(fan_out, fan_in), at + fan_out * fan_in
            x, at = x @ w.t() + p[at:at + fan_out], at + fan_out
            x = torch.nn.functional.silu(x) if fan_out != 3 else x
        keep = mask.bool()
        loss = ((x[keep] - targets[keep][:, :3].double()) ** 2).sum() / int(keep.sum())
        grad, = torch.autograd.grad(loss, p)
        return dict(grad=grad, loss=loss.detach().reshape(1))
    s = _scene(case, seed)
    a, diag, mu = _solution(case, s)
    if kind == "apply":
        out = torch.zeros((s["pos"].shape[0], 4), dtype=torch.float64, device="cuda")
        out[:, :3] = a @ s["vel"][:, :3].double()
        return dict(out=out)
    x = _bicgstab(a, diag, s["b"], s["vel"][:, :3].double())
    if kind == "host":
        return dict(vel=x)
    out = torch.zeros((x.shape[0], 4), dtype=torch.float64, device="cuda")
    out[:, :3] = x
    return dict(vel=out, mu=mu) if case.get("rheology") else dict(vel=out)
