"""The work that users of this framework run on the GPU, as a list of measurable cases.

Every case is one job through the public Python entry points (``Lattice``, ``AdeLattice`` and their
gradient calls): the state is set from fields in device memory, the lattice advances by a few hundred
steps (or runs forward and back for a gradient), and the result is read out.  Kinds:

  ``fluid``    a flow on D2Q9 / D3Q19: initialise, step, read populations, density and velocity
               (with ``stats`` also the lattice statistics of the last collision)
  ``adjoint``  gradient of the plane-mean velocity with respect to the porosity field and tau
  ``force``    gradient of the velocity misfit with respect to the per-cell force field
  ``scalar``   advection-diffusion with a uniform velocity on D2Q5 / D3Q7
  ``coupled``  a fluid and a scalar that it carries, one step of each in turn
"""
import math

import numpy as np
import torch

from paper_2307_11752_gb300 import olb

FLUID, WALL, LID = 1, 2, 3
LID_SPEED = 0.05


def listed():
    return [
        # The smallest job: the guide's 2D Taylor-Green vortex at 64 x 64 in double precision, the set-up of
        # convergence studies.  4096 cells: launches, latency and the FP64 pipe count.
        dict(name="vortex2d_f64_64", kind="fluid", geometry="vortex", nx=64, ny=64, nz=1, dtype="f64",
             scheme="pull", collision="bgk", tau=0.8, steps=500, stats=False),
        # A 2D channel with an obstacle at the size of the guide's bstep2d example (109,291 voxels), body force and
        # porosity, odd extents: an ordinary 2D engineering run, all of it resident in L2.
        dict(name="channel2d_f32_511x213", kind="fluid", geometry="obstacle", nx=511, ny=213, nz=1, dtype="f32",
             scheme="pull", collision="bgk", tau=0.62, steps=400, stats=False, porous=True),
        # A finely resolved 2D lid-driven cavity with statistics, even extents: the largest usual 2D resolution.
        dict(name="cavity2d_f32_1024", kind="fluid", geometry="cavity", nx=1024, ny=1024, nz=1, dtype="f32",
             scheme="pull", collision="bgk", tau=0.55, steps=200, stats=True),
        # The benchmark's lid-driven cavity, two-buffer pull, FP32: the headline workload of this framework.
        dict(name="cavity3d_f32_128", kind="fluid", geometry="cavity", nx=128, ny=128, nz=128, dtype="f32",
             scheme="pull", collision="bgk", tau=0.54725, steps=100, stats=True),
        # The same cavity with 16-bit storage in one buffer (AA): the choice of users short of memory.
        dict(name="cavity3d_f16_aa_128", kind="fluid", geometry="cavity", nx=128, ny=128, nz=128, dtype="f16",
             scheme="aa", collision="bgk", tau=0.54725, steps=100, stats=True),
        # A decaying 3D Taylor-Green vortex far larger than L2, 16-bit storage, every cell fluid and periodic: the
        # largest forward run (turbulence-decay studies).
        dict(name="vortex3d_f16_256", kind="fluid", geometry="vortex", nx=256, ny=256, nz=256, dtype="f16",
             scheme="pull", collision="bgk", tau=0.52, steps=60, stats=False),
        # The forced porous channel of the differentiable workloads, forward only, with the TRT collision that
        # porous-media users choose for its exact wall position.
        dict(name="channel3d_f32_trt_256", kind="fluid", geometry="channel", nx=256, ny=128, nz=128, dtype="f32",
             scheme="pull", collision="trt", tau=0.8, steps=60, stats=False, porous=True),
        # A double-precision 3D channel of ragged extents: reference solutions for validation.
        dict(name="channel3d_f64_75x61x57", kind="fluid", geometry="channel", nx=75, ny=61, nz=57, dtype="f64",
             scheme="pull", collision="bgk", tau=0.7, steps=60, stats=False),
        # One gradient evaluation of porosity identification: checkpointed forward sweep, recompute and adjoint.
        dict(name="adjoint3d_f32_128x64x64", kind="adjoint", nx=128, ny=64, nz=64, dtype="f32", collision="bgk",
             tau=0.8, steps=120, every=20),
        # One gradient evaluation of force-field identification on a small box (launches and host work count).
        dict(name="force3d_f32_48x40x36", kind="force", nx=48, ny=40, nz=36, dtype="f32", collision="bgk", tau=0.7,
             steps=80, every=10),
        # A passive scalar carried by a uniform velocity on a lattice larger than L2.
        dict(name="scalar3d_f32_192", kind="scalar", nx=192, ny=192, nz=192, dtype="f32", walls=False, tau=0.6,
             steps=100),
        # Forced convection: a fluid channel and a scalar with Dirichlet and no-flux walls, coupled at every step.
        dict(name="coupled3d_f32_128x64x60", kind="coupled", nx=128, ny=64, nz=60, dtype="f32", walls=True, tau=0.6,
             fluid_tau=0.7, steps=50),
    ]


def draw(rng):
    """One more job of the same kinds, every extent, option and step count free over its range."""
    def size(lo, hi):
        n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        return n + 1 if n % 2 and rng.random() < 0.5 else n  # three of four even: what users choose most

    kind = rng.choices(["fluid", "adjoint", "force", "scalar", "coupled"], [12, 2, 1, 2, 2])[0]
    tau = round(rng.uniform(0.53, 0.9), 4)
    if kind == "fluid":
        dtype = rng.choices(["f32", "f16", "bf16", "f64"], [5, 3, 1, 2])[0]
        geometry = rng.choice(["vortex", "cavity", "channel", "obstacle"])
        if rng.random() < 0.4:
            nx, ny, nz = size(24, 1400), size(24, 1024), 1
            if dtype == "f64":
                nx, ny = min(nx, 300), min(ny, 300)
            steps = rng.randrange(100, 401)
        else:
            top = {"f64": 80, "f32": 176, "f16": 208, "bf16": 208}[dtype]
            nx, ny, nz = size(20, top), size(20, top), size(20, top)
            steps = rng.randrange(30, 101)
        return dict(kind="fluid", geometry=geometry, nx=nx, ny=ny, nz=nz, dtype=dtype,
                    scheme=rng.choices(["pull", "aa"], [3, 1])[0], collision=rng.choices(["bgk", "trt"], [3, 1])[0],
                    tau=tau, steps=steps, stats=rng.random() < 0.5,
                    porous=geometry in ("channel", "obstacle") and rng.random() < 0.4)
    if kind == "adjoint":
        dtype = rng.choices(["f32", "f16", "f64"], [4, 2, 1])[0]
        top = 48 if dtype == "f64" else 112
        return dict(kind="adjoint", nx=size(24, top), ny=size(20, top), nz=size(16, top), dtype=dtype,
                    collision=rng.choices(["bgk", "trt"], [3, 1])[0], tau=tau, steps=rng.randrange(30, 121),
                    every=rng.randrange(6, 25))
    if kind == "force":
        dtype = rng.choices(["f32", "f64"], [3, 1])[0]
        return dict(kind="force", nx=size(20, 64), ny=size(18, 56), nz=size(16, 56), dtype=dtype, collision="bgk",
                    tau=tau, steps=rng.randrange(20, 81), every=rng.randrange(5, 21))
    if kind == "scalar":
        dtype = rng.choices(["f32", "f64"], [3, 1])[0]
        if rng.random() < 0.35:
            nx, ny, nz = size(32, 1024), size(32, 1024), 1
        else:
            top = 192 if dtype == "f32" else 128
            nx, ny, nz = size(24, top), size(24, top), size(24, top)
        return dict(kind="scalar", nx=nx, ny=ny, nz=nz, dtype=dtype, walls=rng.random() < 0.5, tau=tau,
                    steps=rng.randrange(40, 161))
    nz = 1 if rng.random() < 0.3 else size(16, 112)
    return dict(kind="coupled", nx=size(24, 144), ny=size(20, 112), nz=nz, dtype="f32", walls=True, tau=tau,
                fluid_tau=round(rng.uniform(0.55, 0.9), 4), steps=rng.randrange(20, 81))


# --------------------------------------------------------------------------------------
# Inputs (device tensors, made from the seed alone)
# --------------------------------------------------------------------------------------
def _shape(case):
    return (case["nz"], case["ny"], case["nx"])


def _geometry(case):
    return case.get("geometry", "channel")


def _material(case):
    """Material numbers [nz, ny, nx] and the mask of periodic axes."""
    nz, ny, nx = _shape(case)
    m = torch.full((nz, ny, nx), FLUID, dtype=torch.uint8, device="cuda")
    g = _geometry(case)
    if g == "vortex":
        return m, 7 if nz > 1 else 3
    m[:, 0, :] = WALL
    m[:, -1, :] = WALL
    if nz > 1:
        m[0] = WALL
        m[-1] = WALL
    if g == "cavity":
        m[:, :, 0] = WALL
        m[:, :, -1] = WALL
        m[:, -1, :] = LID
        return m, 0
    if g == "obstacle":  # a cylinder (sphere) behind the inlet, off the centre line
        z, y, x = torch.meshgrid(*[torch.arange(n, device="cuda", dtype=torch.float64) for n in (nz, ny, nx)],
                                 indexing="ij")
        r = 0.15 * min(n for n in (ny, nx, nz) if n > 1)
        d2 = (x - 0.25 * nx) ** 2 + (y - 0.47 * ny) ** 2
        if nz > 1:
            d2 = d2 + (z - 0.5 * nz) ** 2
        m[d2 < r * r] = WALL
    return m, 1


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * (int(seed) + 1))
    return g


def _modes(gen, shape, count, amplitude):
    """A smooth seeded field: ``count`` Fourier modes of low wave number, sup norm at most ``amplitude``."""
    nz, ny, nx = shape
    r = torch.rand((count, 4), generator=gen, device="cuda", dtype=torch.float64)
    out = torch.zeros(shape, device="cuda", dtype=torch.float64)
    axes = [2 * math.pi * torch.arange(n, device="cuda", dtype=torch.float64) / n for n in shape]
    for k in range(count):
        kx, ky, kz = [torch.floor(3.999 * r[k, a]) - 1.0 for a in range(3)]
        out += torch.cos(kz * axes[0][:, None, None] + ky * axes[1][None, :, None] + kx * axes[2][None, None, :]
                         + 2 * math.pi * r[k, 3])
    return out * (amplitude / count)


def _fields(case, gen):
    """Initial density and velocity: the base flow of the geometry plus a seeded smooth disturbance."""
    nz, ny, nx = shape = _shape(case)
    rho = 1.0 + _modes(gen, shape, 3, 1e-3)
    u = torch.stack([_modes(gen, shape, 3, 0.01) for _ in range(3)])
    if nz == 1:
        u[2] = 0.0
    y = 2 * math.pi * torch.arange(ny, device="cuda", dtype=torch.float64) / ny
    x = 2 * math.pi * torch.arange(nx, device="cuda", dtype=torch.float64) / nx
    if _geometry(case) == "vortex":
        u[0] += 0.03 * torch.sin(x)[None, None, :] * torch.cos(y)[None, :, None]
        u[1] -= 0.03 * torch.cos(x)[None, None, :] * torch.sin(y)[None, :, None]
    elif _geometry(case) != "cavity":
        s = (torch.arange(ny, device="cuda", dtype=torch.float64) - 0.5) / (ny - 2)
        u[0] += (0.16 * s * (1 - s)).clamp(min=0.0)[None, :, None]
    return rho, u


def _porosity(gen, shape):
    """Porosity in [0, 1]: mostly open, with smooth resistive patches."""
    return (0.85 + _modes(gen, shape, 4, 0.6)).clamp(0.0, 1.0)


def _body_force(case):
    """The force that keeps a plane channel of this height at a centre speed of 0.04."""
    if _geometry(case) in ("vortex", "cavity"):
        return (0.0, 0.0, 0.0)
    nu = (case.get("fluid_tau", case["tau"]) - 0.5) / 3.0
    return (8.0 * nu * 0.04 / (case["ny"] - 2) ** 2, 0.0, 0.0)


def _inputs(case, seed):
    gen = _generator(seed)
    d = dict(case=dict(case), shape=_shape(case))
    if case["kind"] != "scalar":
        d["material"], d["periodic"] = _material(case)
        d["rho"], d["u"] = _fields(case, gen)
        d["force"] = _body_force(case)
        d["gamma"] = _porosity(gen, d["shape"]) if case.get("porous") or case["kind"] == "adjoint" else None
    if case["kind"] == "force":
        d["force_field"] = torch.stack([_modes(gen, d["shape"], 4, 2e-5) for _ in range(3)])
        d["force_field"][0] += d["force"][0]
        d["target"] = d["u"] * 0.9
    if case["kind"] in ("scalar", "coupled"):
        d["C"] = 0.5 + _modes(gen, d["shape"], 4, 0.4)
        d["velocity"] = (0.04, -0.02, 0.03 if case["nz"] > 1 else 0.0)
        d["scalar_material"], d["scalar_periodic"], d["wall_C"] = _scalar_walls(case)
    return d


def _scalar_walls(case):
    """Hot and cold plates on the y faces (Dirichlet), insulating z faces, periodic x; or no walls at all."""
    if not case["walls"]:
        return None, 7 if case["nz"] > 1 else 3, None
    m = torch.ones(_shape(case), dtype=torch.uint8, device="cuda")
    if case["nz"] > 1:
        m[0] = 0
        m[-1] = 0
    m[:, 0, :] = 2
    m[:, -1, :] = 3
    return m, 1, [0.0, 0.0, 1.0, 0.0]


# --------------------------------------------------------------------------------------
# The calls
# --------------------------------------------------------------------------------------
def _lattice(case, d, dtype, scheme, tau):
    nz, ny, nx = d["shape"]
    lat = olb.Lattice(olb.D3Q19 if nz > 1 else olb.D2Q9, (nx, ny, nz), dtype=dtype, scheme=scheme)
    lat.set_material(d["material"], d["periodic"])
    lat.set_wall_velocity(LID, (LID_SPEED, 0.0, 0.0))
    if case.get("collision") == "trt":
        lat.set_trt(tau, 3.0 / 16.0)
    else:
        lat.set_bgk(tau)
    lat.set_force(d["force"])
    if d["gamma"] is not None:
        lat.set_porosity(d["gamma"])
    return lat


def prepare(case, seed):
    d = _inputs(case, seed)
    kind = case["kind"]
    if kind != "scalar":
        tau = case.get("fluid_tau", case["tau"])
        d["lattice"] = _lattice(case, d, case["dtype"], case.get("scheme", "pull"), tau)
    if kind in ("adjoint", "force"):
        d["lattice"].init_equilibrium(d["rho"], d["u"])
        d["f0"] = d["lattice"].get_populations()
    if kind in ("scalar", "coupled"):
        nz, ny, nx = d["shape"]
        a = olb.AdeLattice(olb.D3Q7 if nz > 1 else olb.D2Q5, (nx, ny, nz), case["dtype"])
        a.set_tau(case["tau"])
        a.set_velocity(d["velocity"])
        if d["scalar_material"] is not None:
            a.set_material(d["scalar_material"], d["scalar_periodic"], d["wall_C"])
        d["scalar"] = a
    return d


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "fluid":
        lat, out = state["lattice"], {}
        lat.init_equilibrium(state["rho"], state["u"])
        if case["stats"]:
            out["stats"] = lat.step_stats(case["steps"])
        else:
            lat.step(case["steps"])
        out["rho"], out["u"] = lat.moments()
        out["f"] = lat.get_populations()
        return out
    if kind == "adjoint":
        gamma = state["gamma"].detach().requires_grad_(True)
        tau = torch.tensor(case["tau"], dtype=torch.float64, requires_grad=True)
        lat = state["lattice"]
        if case["collision"] == "trt":  # the autograd wrapper selects BGK; TRT users call the lattice itself
            lat.set_porosity(state["gamma"])
            lat.set_populations(state["f0"])
            loss, dgamma, dtau = lat.adjoint_run(case["steps"], case["every"], (0, case["nx"] - 1, 0))
            return {"loss": loss, "dgamma": dgamma, "dtau": dtau}
        loss = olb.plane_velocity_loss(lat, gamma, tau, state["f0"], case["steps"], case["every"],
                                       (0, case["nx"] - 1, 0))
        loss.backward()
        return {"loss": loss.detach(), "dgamma": gamma.grad, "dtau": tau.grad}
    if kind == "force":
        F = state["force_field"].detach().requires_grad_(True)
        loss = olb.force_misfit_loss(state["lattice"], F, state["f0"], case["steps"], case["every"], state["target"])
        loss.backward()
        return {"loss": loss.detach(), "dforce": F.grad}
    a = state["scalar"]
    if kind == "scalar":
        a.init(state["C"])
        a.step(case["steps"])
        return {"C": a.density()}
    fluid = state["lattice"]
    fluid.init_equilibrium(state["rho"], state["u"])
    a.set_velocity_from(fluid)
    a.init(state["C"])
    for _ in range(case["steps"]):
        fluid.step(1)
        a.set_velocity_from(fluid)
        a.step(1)
    rho, u = fluid.moments()
    return {"C": a.density(), "rho": rho, "u": u}


def work(case):
    """Inputs read once and outputs written once; the arithmetic of every cell update."""
    cells = case["nx"] * case["ny"] * case["nz"]
    three = case["nz"] > 1
    q, qs = (19, 7) if three else (9, 5)
    fluid_flops, scalar_flops = (250, 40) if three else (110, 28)
    kind, n = case["kind"], case["steps"]
    if kind == "fluid":
        fields = 4 + (1 if case.get("porous") else 0)  # rho, u (and porosity) in
        return {"bytes": cells * 8 * (fields + 4 + q), "flops": cells * n * fluid_flops}
    if kind == "adjoint":  # forward, recompute and about twice a step's arithmetic for the adjoint
        return {"bytes": cells * 8 * (q + 2), "flops": cells * n * 4 * fluid_flops}
    if kind == "force":
        return {"bytes": cells * 8 * (q + 9), "flops": cells * n * 4 * fluid_flops}
    if kind == "scalar":
        return {"bytes": cells * 8 * 2, "flops": cells * n * scalar_flops}
    return {"bytes": cells * 8 * (4 + 1 + 4 + 1), "flops": cells * n * (fluid_flops + scalar_flops)}


# --------------------------------------------------------------------------------------
# The same results from plain torch in 64 bits
# --------------------------------------------------------------------------------------
_C9 = [(0, 0, 0), (-1, 1, 0), (-1, 0, 0), (-1, -1, 0), (0, -1, 0), (1, -1, 0), (1, 0, 0), (1, 1, 0), (0, 1, 0)]
_HALF19 = [(-1, 0, 0), (0, -1, 0), (0, 0, -1), (-1, -1, 0), (-1, 1, 0), (-1, 0, -1), (-1, 0, 1), (0, -1, -1),
           (0, -1, 1)]
_C19 = [(0, 0, 0)] + _HALF19 + [tuple(-a for a in c) for c in _HALF19]


def _shift(a, c):
    """b(x) = a(x - c), wrapped; the last three axes are z, y, x."""
    return torch.roll(a, (c[2], c[1], c[0]), (-3, -2, -1)) if any(c) else a


def _blocked(open_cells, periodic, c):
    """True where x + c is not an open cell (or lies outside along an axis that does not wrap)."""
    ok = _shift(open_cells, tuple(-a for a in c)).clone()
    for axis, a in enumerate(c):
        if a and not periodic & (1 << axis):
            ok.select(2 - axis, -1 if a > 0 else 0).fill_(False)
    return ~ok


class _Flow:
    def __init__(self, d):
        case, m = d["case"], d["material"]
        self.c = _C19 if case["nz"] > 1 else _C9
        self.w = [{0: 4 / 9, 1: 1 / 9, 2: 1 / 36} if case["nz"] == 1 else {0: 1 / 3, 1: 1 / 18, 2: 1 / 36}][0]
        self.w = [self.w[sum(abs(a) for a in c)] for c in self.c]
        self.opp = [self.c.index(tuple(-a for a in c)) for c in self.c]
        self.fluid = m == FLUID
        lid = m == LID
        self.blocked = [_blocked(self.fluid, d["periodic"], c) for c in self.c]
        # density factor of the population that returns along -c_i from a moving wall
        self.lid = [torch.where(self.blocked[i] & _shift(lid, tuple(-a for a in c)), 6 * self.w[i] * c[0] * LID_SPEED,
                                0.0) for i, c in enumerate(self.c)]
        if not bool(lid.any()):
            self.lid = None
        self.trt = case.get("collision") == "trt"

    def equilibrium(self, rho, u):
        usq = (u * u).sum(0)
        f = []
        for c, w in zip(self.c, self.w):
            cu = sum(a * u[k] for k, a in enumerate(c) if a)
            f.append(w * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * usq))
        return torch.stack(f)

    def moments(self, f, F):
        rho = f.sum(0)
        j = [sum(c[a] * f[i] for i, c in enumerate(self.c) if c[a]) + torch.zeros_like(rho) for a in range(3)]
        return rho, torch.stack([(j[a] + 0.5 * F[a]) / rho for a in range(3)])

    def step(self, f, tau, F, gamma):
        rho, u = self.moments(f, F)
        up = u if gamma is None else gamma * u
        feq = self.equilibrium(rho, up)
        om = 1.0 / tau
        om_odd = 1.0 / ((3.0 / 16.0) / (tau - 0.5) + 0.5) if self.trt else om
        uF = sum(up[a] * F[a] for a in range(3))
        post = []
        for i, (c, w) in enumerate(zip(self.c, self.w)):
            o = self.opp[i]
            even, odd = 0.5 * (f[i] - feq[i] + f[o] - feq[o]), 0.5 * (f[i] - feq[i] - f[o] + feq[o])
            cu = sum(c[a] * up[a] for a in range(3))
            cF = sum(c[a] * F[a] for a in range(3))
            post.append(f[i] - om * even - om_odd * odd + (1 - 0.5 * om) * w * (9 * cu * cF - 3 * uF)
                        + (1 - 0.5 * om_odd) * w * 3 * cF)
        new = []
        for i, c in enumerate(self.c):
            o = self.opp[i]
            back = post[o] if self.lid is None else post[o] - rho * self.lid[o]
            v = torch.where(self.blocked[o], back, _shift(post[i], c)) if any(c) else post[i]
            new.append(torch.where(self.fluid, v, self.w[i]))
        return torch.stack(new)

    def shown(self, a):
        return torch.where(self.fluid, a, 0.0)

    def statistics(self, f, F):
        rho, u = self.moments(f, F)
        uu = (u * u).sum(0)
        k = self.fluid
        j = [sum(c[a] * f[i] for i, c in enumerate(self.c) if c[a]) + torch.zeros_like(rho) for a in range(3)]
        return np.array([float(rho[k].sum())] + [float(j[a][k].sum()) for a in range(3)]
                        + [float(0.5 * uu[k].sum()), float(uu[k].max().sqrt()), 0.0])


class _Scalar:
    def __init__(self, d):
        case = d["case"]
        faces = [(-1, 0, 0), (0, -1, 0), (0, 0, -1), (1, 0, 0), (0, 1, 0), (0, 0, 1)]
        self.c = [(0, 0, 0)] + [c for c in faces if case["nz"] > 1 or c[2] == 0]
        self.cs2 = 0.25 if case["nz"] > 1 else 1 / 3
        self.w = [0.25] + [0.125] * 6 if case["nz"] > 1 else [1 / 3] + [1 / 6] * 4
        self.opp = [self.c.index(tuple(-a for a in c)) for c in self.c]
        m = d["scalar_material"]
        if m is None:
            m = torch.ones(d["shape"], dtype=torch.uint8, device="cuda")
        self.bulk = m == 1
        self.blocked = [_blocked(self.bulk, d["scalar_periodic"], c) for c in self.c]
        self.held, self.value = [], []
        table = torch.zeros(256, dtype=torch.float64, device="cuda")
        if d["wall_C"] is not None:
            table[:len(d["wall_C"])] = torch.tensor(d["wall_C"], dtype=torch.float64)
        for c in self.c:
            n = _shift(m, tuple(-a for a in c))
            outside = _blocked(torch.ones_like(self.bulk), d["scalar_periodic"], c)
            self.held.append((n >= 2) & ~outside)
            self.value.append(table[n.long()])

    def equilibrium(self, C, v):
        return torch.stack([w * C * (1 + sum(c[a] * v[a] for a in range(3)) / self.cs2)
                            for c, w in zip(self.c, self.w)])

    def step(self, g, tau, v):
        post = g - (g - self.equilibrium(g.sum(0), v)) / tau
        new = []
        for i, c in enumerate(self.c):
            o = self.opp[i]
            back = torch.where(self.held[o], -post[o] + 2 * self.w[o] * self.value[o], post[o])
            v_in = torch.where(self.blocked[o], back, _shift(post[i], c)) if any(c) else post[i]
            new.append(torch.where(self.bulk, v_in, g[i]))
        return torch.stack(new)


def _gradients(flow, d, case):
    """Reverse mode of the plain steps, each step recomputed on the way back."""
    from torch.utils.checkpoint import checkpoint

    tau = torch.tensor(case["tau"], dtype=torch.float64, device="cuda", requires_grad=True)
    if case["kind"] == "adjoint":
        gamma = d["gamma"].clone().requires_grad_(True)
        F = torch.tensor(d["force"], dtype=torch.float64, device="cuda")
    else:
        gamma, F = None, d["force_field"].clone().requires_grad_(True)
    f = flow.equilibrium(d["rho"], d["u"])
    f = torch.where(flow.fluid, f, torch.tensor(flow.w, dtype=torch.float64, device="cuda")[:, None, None, None])
    for _ in range(case["steps"]):
        f = checkpoint(flow.step, f, tau, F, gamma, use_reentrant=False)
    rho, u = flow.moments(f, F)
    if case["kind"] == "adjoint":
        plane = flow.fluid[:, :, case["nx"] - 1]
        loss = u[0, :, :, case["nx"] - 1][plane].sum() / plane.sum()
        dg, dtau = torch.autograd.grad(loss, (gamma, tau))
        return {"loss": loss.detach(), "dgamma": dg, "dtau": dtau}
    e = torch.where(flow.fluid, u - d["target"], 0.0)
    loss = 0.5 * (e * e).sum()
    return {"loss": loss.detach(), "dforce": torch.autograd.grad(loss, F)[0]}


def exact(case, seed):
    cells, n = case["nx"] * case["ny"] * case["nz"], case["steps"]
    if cells * n > 4e8 or (case["kind"] in ("adjoint", "force") and cells * n > 8e7):
        return None
    d, kind = _inputs(case, seed), case["kind"]
    if kind in ("adjoint", "force"):
        return _gradients(_Flow(d), d, case)
    with torch.no_grad():
        if kind == "fluid":
            flow, out = _Flow(d), {}
            f = flow.equilibrium(d["rho"], d["u"])
            f = torch.where(flow.fluid, f, 1.0 / len(flow.c))
            for s in range(n):
                if case["stats"] and s == n - 1:
                    out["stats"] = flow.statistics(f, d["force"])
                f = flow.step(f, case["tau"], d["force"], d["gamma"])
            rho, u = flow.moments(f, d["force"])
            out.update(rho=flow.shown(rho), u=flow.shown(u), f=flow.shown(f))
            return out
        scalar = _Scalar(d)
        if kind == "scalar":
            g = scalar.equilibrium(d["C"], d["velocity"])
            for _ in range(n):
                g = scalar.step(g, case["tau"], d["velocity"])
            return {"C": g.sum(0)}
        flow = _Flow(d)
        f = torch.where(flow.fluid, flow.equilibrium(d["rho"], d["u"]), 1.0 / len(flow.c))
        v = flow.shown(flow.moments(f, d["force"])[1])
        g = scalar.equilibrium(d["C"], v)
        for _ in range(n):
            f = flow.step(f, case["fluid_tau"], d["force"], None)
            v = flow.shown(flow.moments(f, d["force"])[1])
            g = scalar.step(g, case["tau"], v)
        rho, u = flow.moments(f, d["force"])
        return {"C": g.sum(0), "rho": flow.shown(rho), "u": flow.shown(u)}
