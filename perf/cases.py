"""The workloads on which the speed of this framework is measured.

A case is one short solve as a user's program runs it: the handles (and the
batch over them) exist, `run` sets the initial droplets, takes the time steps
and reads the fields back. `exact` repeats the solve in 64 bits with plain
torch operations, one line of the method per statement and none of the
framework's code.

Kinds of case
  one    one 2D lattice (``Solver``): init_droplet, step, get_device, and for
         contact-angle studies mass and contact_angle
  batch  several 2D lattices advanced together (``Batch``)
  box    one 3D lattice (``Solver3D``): init_droplet, step, get_f32 into
         pinned host arrays (the 3D read-back is a host call)

The solves are kept short; a real one takes 1,000 to 20,000 steps.
Geometry, lattice sizes and parameters are those of the framework's workloads
(contact-angle cases, many-droplet lattice, uneven batch, request stream, width
sweep, 3D box), and `draw` takes sizes between and beside them, odd ones among
them. The seed decides the droplets' places and radii and the contact angles.
"""
import math

import numpy as np
import torch

from paper_2312_00369_gb300 import pflbm, workloads

_BYTES = {"fp64": 8, "fp32": 4, "bf16": 2, "fp16": 2}


def listed():
    return [
        # contact-angle study on a flat wall in the parity precision: the
        # smallest lattice anyone runs, where the latency of a step is all
        dict(name="flat_100x50_fp64", kind="one", shape="flat", nx=100, ny=50, precision="fp64", steps=400,
             angle=True),
        # the paper's flat-wall table (256 x 128, R = 50, nu = 0.1, M = 0.01)
        dict(name="flat_256x128_fp32", kind="one", shape="flat", nx=256, ny=128, precision="fp32", steps=400,
             sigma=0.005, M=0.01, rho_l=10.0, rho_g=1.0, angle=True),
        # droplet on a staircase wall and on a cylinder: the geometry studies,
        # which leave the (1/2) dG/dt term out so that long runs stay stable
        dict(name="incline_400x200_fp32", kind="one", shape="incline", nx=400, ny=200, precision="fp32", steps=400,
             dgdt=1, angle=True),
        dict(name="cylinder_512x512_fp32", kind="one", shape="cylinder", nx=512, ny=512, precision="fp32", steps=200,
             dgdt=1, angle=True),
        # odd sizes with an angle field, phi-dependent viscosity and gravity
        dict(name="many_1021x383_visc_fp32", kind="one", shape="many", nx=1021, ny=383, precision="fp32", steps=100,
             drops=8, nu_l=0.3, nu_g=0.05, gx=2e-6, gy=-1e-6),
        # the headline lattice: 64 droplets, an angle per droplet
        dict(name="many_4096x2048_fp32", kind="one", shape="many", nx=4096, ny=2048, precision="fp32", steps=100,
             drops=64),
        dict(name="many_4096x2048_bf16", kind="one", shape="many", nx=4096, ny=2048, precision="bf16", steps=100,
             drops=64),
        # 256 independent solves of four sizes and three wall types
        dict(name="batch_256_bf16", kind="batch", mix="uneven", count=256, precision="bf16", steps=200),
        # one tick of the request server: the residents' next 200 steps
        dict(name="serve_16_fp16", kind="batch", mix="requests", count=16, precision="fp16", steps=200, dgdt=1),
        # interface-width sweep: W = 4, 6, 8 at two angles on a shallow staircase
        dict(name="wsweep_6x256x256_fp32", kind="batch", mix="wsweep", count=6, precision="fp32", steps=200, dgdt=1),
        # 3D contact angle on a flat wall
        dict(name="flat_96x96x56_fp32", kind="box", nx=96, ny=96, nz=56, precision="fp32", steps=200, drops=1, dgdt=1),
        # the 3D headline box
        dict(name="many_512x512x128_fp32", kind="box", nx=512, ny=512, nz=128, precision="fp32", steps=40, drops=64),
    ]


def _log_between(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["one", "one", "one", "batch", "box"])
    dgdt = rng.choice([0, 1])
    if kind == "box":
        precision = rng.choice(["fp32", "fp32", "fp32", "fp64"])
        nx, ny, nz = _log_between(rng, 24, 320), _log_between(rng, 24, 320), _log_between(rng, 20, 120)
        most = (1.5e9 if precision == "fp32" else 5e7) / (nx * ny * nz)
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, precision=precision, dgdt=dgdt,
                    drops=rng.randint(1, 8), steps=max(4, min(_log_between(rng, 20, 200), int(most))))
    precision = rng.choice(["fp32", "fp32", "bf16", "fp16", "fp64"])
    slow = 14.0 if precision == "fp64" else 1.0
    if kind == "batch":
        mix = rng.choice(["uneven", "requests", "wsweep"])
        count = {"uneven": _log_between(rng, 4, 128), "requests": _log_between(rng, 2, 16),
                 "wsweep": rng.randint(2, 6)}[mix]
        most = 8e8 / slow / (count * {"uneven": 41e3, "requests": 130e3, "wsweep": 66e3}[mix])
        return dict(kind=kind, mix=mix, count=count, precision=precision, dgdt=dgdt,
                    steps=max(8, min(_log_between(rng, 50, 400), int(most))))
    shape = rng.choice(["flat", "incline", "cylinder", "many"])
    nodes = math.exp(rng.uniform(math.log(5e3), math.log(8.3e6 if shape == "many" else 1e6)))
    aspect = {"flat": 2.0, "incline": 2.0, "cylinder": 1.0, "many": 2.0}[shape] * math.exp(rng.uniform(-0.2, 0.2))
    ny = max(48, int(round(math.sqrt(nodes / aspect))))
    nx = max(49, int(round(nodes / ny)))
    case = dict(kind=kind, shape=shape, nx=nx, ny=ny, precision=precision, dgdt=dgdt,
                steps=max(4, min(_log_between(rng, 20, 400), int(8e8 / slow / (nx * ny)))))
    if shape == "many":
        case["drops"] = max(1, nx // 64)
    else:
        case["angle"] = bool(rng.getrandbits(1))
    if rng.random() < 0.3:
        case.update(nu_l=rng.uniform(0.1, 0.3), nu_g=rng.uniform(0.05, 0.1), gx=rng.uniform(-2e-6, 2e-6),
                    gy=rng.uniform(-2e-6, 0.0))
    return case


# ---------------------------------------------------------------------------
# what a case holds: lattices with their droplets, angles and parameters
# ---------------------------------------------------------------------------

def _geometry(shape, nx, ny):
    """(solid, wall, droplet centre, droplet radius) of a 2D lattice."""
    if shape in ("flat", "many"):
        solid, wall = workloads.flat_channel(nx, ny)
        return solid, wall, (nx / 2.0, wall["py"]), 0.4 * ny
    if shape == "incline":
        solid, wall = workloads.inclined(nx, ny, 30.0)
        return solid, wall, (nx / 2.0, math.tan(math.radians(30.0)) * nx / 2.0), ny / 5.0
    if shape == "shallow":
        solid, wall = workloads.inclined(nx, ny, math.degrees(math.atan(0.25)))
        return solid, wall, (nx / 2.0, nx / 8.0), ny / 5.0
    radius = ny / 5.0 if shape == "cylinder" else ny / 4.0          # "low_cylinder": the batch's
    centre = (nx / 2.0, ny / 2.0 if shape == "cylinder" else 0.4 * ny)
    solid, wall = workloads.cylinder(nx, ny, centre[0], centre[1], radius)
    return solid, wall, (centre[0], centre[1] + radius), (ny / 10.0 if shape == "cylinder" else ny / 5.0)


def _lattice(case, shape, nx, ny, rng, W=4.0):
    solid, wall, centre, radius = _geometry(shape, nx, ny)
    lat = dict(solid=solid, wall=wall, W=W, theta=float(rng.uniform(30.0, 150.0)), field=None)
    if shape == "many":
        n = case["drops"]
        r = rng.uniform(30.0, 60.0, n) * min(1.0, ny / 150.0)
        xs, angles = rng.uniform(0.0, nx, n), rng.uniform(30.0, 150.0, n)
        lat["drops"] = [(float(x), centre[1], float(q)) for x, q in zip(xs, r)]
        far = np.abs(np.arange(nx)[:, None] - xs[None, :])
        nearest = angles[np.argmin(np.minimum(far, nx - far), axis=1)]
        lat["field"] = np.ascontiguousarray(np.broadcast_to(nearest[None, :], (ny, nx)).astype(np.float32))
    else:
        lat["drops"] = [(centre[0] + float(rng.uniform(-2, 2)), centre[1], radius * float(rng.uniform(0.9, 1.1)))]
    return lat


def _sizes(case):
    """(shape, nx, ny, W) of every lattice of a batch, from the case alone."""
    n = case["count"]
    if case["mix"] == "wsweep":
        return [("shallow", 256, 256, (4.0, 6.0, 8.0)[k % 3]) for k in range(n)]
    shapes = ("flat", "incline", "low_cylinder")
    if case["mix"] == "uneven":
        rng = np.random.default_rng(369)
        return [(shapes[int(rng.integers(3))], *workloads.BATCH_SIZES[int(rng.integers(4))], 4.0) for _ in range(n)]
    stream = workloads.request_stream(n_max=n)
    return [(shapes[d["wall_type"]], d["nx"], d["ny"], 4.0) for d in stream]


def _lattices(case, seed):
    rng = np.random.default_rng(seed)
    if case["kind"] == "one":
        return [_lattice(case, case["shape"], case["nx"], case["ny"], rng)]
    return [_lattice(case, shape, nx, ny, rng, W) for shape, nx, ny, W in _sizes(case)]


def _box(case, seed):
    rng = np.random.default_rng(seed)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    solid, zw = workloads.box3d(nx, ny, nz)
    r = rng.uniform(12.0, 24.0, case["drops"]) * min(1.0, nz / 50.0)
    drops = [(float(rng.uniform(0, nx)), float(rng.uniform(0, ny)), zw, float(q)) for q in r]
    return dict(solid=solid, drops=drops, W=4.0, theta=float(rng.uniform(40.0, 120.0)), field=None)


def _physics(case):
    p = dict(sigma=0.01, M=0.1, tau_f=0.8, rho_l=1.0, rho_g=0.1)
    p.update({k: case[k] for k in ("sigma", "M", "rho_l", "rho_g") if k in case})
    return p


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------

_STREAM = []


def _stream():
    """The program's one work stream (members of a batch have to share one,
    and it must not be the default stream)."""
    if not _STREAM:
        _STREAM.append(torch.cuda.Stream())
    return _STREAM[0]


def prepare(case, seed):
    common = dict(_physics(case), precision=case["precision"], dgdt_mode=case.get("dgdt", 0), stream=_stream())
    if case["kind"] == "box":
        lat = _box(case, seed)
        solver = pflbm.Solver3D(lat["solid"], theta_deg=lat["theta"], W=lat["W"], **common)
        shape = lat["solid"].shape
        out = [torch.empty(s, dtype=torch.float32).pin_memory() for s in (shape, shape + (3,), shape)]
        return dict(kind="box", solver=solver, drops=lat["drops"], steps=case["steps"],
                    out=tuple(t.numpy() for t in out), pinned=out)
    common.update({k: case[k] for k in ("nu_l", "nu_g", "gx", "gy") if k in case})
    lats = _lattices(case, seed)
    solvers = [pflbm.Solver(lat["solid"], theta_deg=lat["theta"], theta_field=lat["field"], W=lat["W"], **common)
               for lat in lats]
    # one buffer per field over all lattices; each lattice fills its own part
    ends = np.cumsum([s.nx * s.ny for s in solvers])
    phi, u, p = (torch.empty(int(ends[-1]) * c, dtype=torch.float64, device="cuda") for c in (1, 2, 1))
    parts = [(phi[e - s.nx * s.ny:e], u[2 * (e - s.nx * s.ny):2 * e], p[e - s.nx * s.ny:e])
             for s, e in zip(solvers, ends.tolist())]
    state = dict(kind=case["kind"], solvers=solvers, drops=[lat["drops"] for lat in lats], steps=case["steps"],
                 out=(phi, u, p), parts=parts, wall=lats[0]["wall"] if case.get("angle") else None)
    if case["kind"] == "batch":
        state["batch"] = pflbm.Batch(solvers)
    return state


def run(state):
    if state["kind"] == "box":
        solver = state["solver"]
        for drop in state["drops"]:
            solver.init_droplet(*drop)
        solver.step(state["steps"])
        return dict(zip(("phi", "u", "p"), solver.get_f32(state["out"])))
    for solver, drops in zip(state["solvers"], state["drops"]):
        for drop in drops:
            solver.init_droplet(*drop)
    (state["batch"] if state["kind"] == "batch" else state["solvers"][0]).step(state["steps"])
    for solver, part in zip(state["solvers"], state["parts"]):
        solver.get_device(*part)
    torch.cuda.current_stream().wait_stream(_stream())      # whoever reads the fields next
    out = dict(zip(("phi", "u", "p"), state["out"]))
    if state["wall"] is not None:
        out["mass"] = state["solvers"][0].mass()
        out["angle"] = state["solvers"][0].contact_angle(state["wall"])[0]
    return out


def work(case):
    """The state after the last step and the fields, written once, and the
    node bytes, read once; the arithmetic of every step on the non-solid
    nodes. (A step's populations need not pass through HBM.)"""
    e = _BYTES[case["precision"]]
    if case["kind"] == "box":
        nodes, fluid = (case["nx"] * case["ny"] * d for d in (case["nz"], case["nz"] - 4))
        return {"bytes": nodes * (1 + 20) + fluid * 26 * e, "flops": 410 * fluid * case["steps"]}
    sizes = [(case["shape"], case["nx"], case["ny"], 4.0)] if case["kind"] == "one" else _sizes(case)
    nodes = sum(nx * ny for _, nx, ny, _ in sizes)
    fluid = sum(int((_geometry(shape, nx, ny)[0] == 0).sum()) for shape, nx, ny, _ in sizes)
    # 16-bit states keep g_0 in 32 bits
    return {"bytes": nodes * (1 + 32) + fluid * (18 * e + (2 if e == 2 else 0)),
            "flops": 228 * fluid * case["steps"]}


# ---------------------------------------------------------------------------
# the method in 64 bits, on [..., ny, nx] or [..., nz, ny, nx] fields
# ---------------------------------------------------------------------------

_AXES2 = [(1, 0), (0, 1)]
_C2 = [(0, 0)] + [(s * a, s * b) for a, b in _AXES2 for s in (1, -1)] + [(s, t) for s in (1, -1) for t in (1, -1)]
_C3G = [(0, 0, 0)] + [tuple(s * (d == k) for k in range(3)) for d in range(3) for s in (1, -1)]
_C3F = _C3G + [c for d in range(3) for c in
               [tuple(s if k == (d + 1) % 3 else t if k == (d + 2) % 3 else 0 for k in range(3))
                for s in (1, -1) for t in (1, -1)]]


class _Lattice:
    """Velocities (x first), weights, opposites and c_s^2."""

    def __init__(self, c, weight, cs2):
        self.c, self.cs2 = c, cs2
        self.w = [weight[sum(abs(k) for k in v)] for v in c]
        self.opp = [c.index(tuple(-k for k in v)) for v in c]


def _moved(a, c):
    """a(x - c). What wraps around in the wall-normal axis (y in 2D, z in 3D)
    lands in solid rows that no fluid node reads."""
    if not any(c):
        return a
    return torch.roll(a, shifts=tuple(c), dims=tuple(-1 - k for k in range(len(c))))


class _Reference:
    """The scheme of the paper in 64 bits: moments, collisions, streaming and
    the modified bounce-back, each over the whole field."""

    def __init__(self, solid, theta, W, case):
        ph = _physics(case)
        dim = 3 if case["kind"] == "box" else 2
        if dim == 2:
            self.F = self.G = _Lattice(_C2, {0: 4 / 9, 1: 1 / 9, 2: 1 / 36}, 1 / 3)
        else:
            self.F = _Lattice(_C3F, {0: 1 / 3, 1: 1 / 18, 2: 1 / 36}, 1 / 3)
            self.G = _Lattice(_C3G, {0: 1 / 4, 1: 1 / 8}, 1 / 4)
        self.dim, self.W, self.dgdt = dim, W, case.get("dgdt", 0)
        self.beta, self.kappa = 12 * ph["sigma"] / W, 1.5 * ph["sigma"] * W
        self.alpha = ph["M"] / (self.G.cs2 * 0.5)               # tau_g = 1
        self.tau, self.rho_g, self.drho = ph["tau_f"], ph["rho_g"], ph["rho_l"] - ph["rho_g"]
        self.nu = (case["nu_l"], case["nu_g"]) if "nu_l" in case else None
        self.body = (case.get("gx", 0.0), case.get("gy", 0.0), 0.0)[:dim]
        # node classes: fluid, boundary (solid beside fluid), ghost, interior
        steps = self.F.c[1:]
        beside = torch.zeros_like(solid)
        for c in steps:
            beside |= ~_moved(solid, c)
        self.zeta = ~solid | beside
        near = torch.zeros_like(solid)
        for c in steps:
            near |= _moved(self.zeta, c)
        self.ghost = ~self.zeta & near
        # a ghost node's neighbours: the whole 3^dim - 1 block
        self.block = [c for c in np.ndindex(*(3,) * dim)]
        self.block = [tuple(int(k) - 1 for k in c) for c in self.block if any(k != 1 for k in c)]
        self.near = sum(_moved(self.zeta, c).double() for c in self.block).clamp(min=1.0)
        eps_grad, _ = self.stencil((~solid).double())
        av = torch.sqrt(sum(g * g for g in eps_grad))
        self.wet = av * math.sqrt(2 * self.kappa * self.beta) * torch.cos(theta * (math.pi / 180))
        self.known = [_moved(self.zeta, c) for c in self.F.c]

    def stencil(self, v):
        L, grad, lap = self.F, [0.0] * self.dim, 0.0
        for c, w in zip(L.c[1:], L.w[1:]):
            at = _moved(v, tuple(-k for k in c))
            for d in range(self.dim):
                if c[d]:
                    grad[d] = grad[d] + (w * c[d] / L.cs2) * at
            lap = lap + (2 * w / L.cs2) * (at - v)
        return grad, lap

    def droplets(self, drops):
        """0.5 + 0.5 tanh(2 (R - r) / W), the largest over the droplets; the
        wall-normal axis is the only one that is not periodic."""
        phi = torch.zeros_like(self.near)
        grid = [torch.arange(n, dtype=torch.float64, device=phi.device) for n in phi.shape[-self.dim:]]
        coords = torch.meshgrid(*grid, indexing="ij")[::-1]      # x first
        for drop in drops:                                       # per lattice of the stack
            r2 = 0.0
            for d in range(self.dim):
                at = torch.as_tensor([q[d] for q in drop], dtype=torch.float64, device=phi.device)
                delta = coords[d] - at.reshape((-1,) + (1,) * self.dim)
                if d < self.dim - 1:
                    n = phi.shape[-1 - d]
                    delta = delta - n * torch.round(delta / n)
                r2 = r2 + delta * delta
            R = torch.as_tensor([q[-1] for q in drop], dtype=torch.float64, device=phi.device)
            v = 0.5 + 0.5 * torch.tanh(2 * (R.reshape((-1,) + (1,) * self.dim) - torch.sqrt(r2)) / self.W)
            phi = torch.maximum(phi, v)
        self.phi = torch.where(self.zeta, phi, 0.0)
        self.potential()
        self.f = [torch.zeros_like(phi) for _ in self.F.c]
        self.g = [w * self.alpha * self.mu for w in self.G.w]
        self.g[0] = self.phi - (1 - self.G.w[0]) * self.alpha * self.mu
        self.last = None

    def potential(self):
        """Ghost values, gradients and the chemical potential from phi."""
        total = sum(_moved(torch.where(self.zeta, self.phi, 0.0), c) for c in self.block)
        self.phi = torch.where(self.ghost, total / self.near, torch.where(self.zeta, self.phi, 0.0))
        self.grad, lap = self.stencil(self.phi)
        q = self.phi
        self.mu = 4 * self.beta * q * (q - 1) * (q - 0.5) - self.kappa * lap - self.wet * (q - q * q)

    def moments(self):
        L = self.F
        self.phi = sum(self.g)
        self.potential()
        self.rho = self.phi * self.drho + self.rho_g
        self.force = [self.mu * g + self.rho * b for g, b in zip(self.grad, self.body)]
        self.u = []
        for d in range(self.dim):
            m = sum(c[d] * f for c, f in zip(L.c, self.f) if c[d])
            self.u.append((m + 0.5 * self.force[d]) / self.rho)
        self.uu = sum(u * u for u in self.u)
        self.urho = self.drho * sum(u * g for u, g in zip(self.u, self.grad))
        s0 = -L.w[0] * self.uu / (2 * L.cs2)
        self.p = L.cs2 / (1 - L.w[0]) * (sum(self.f[1:]) + 0.5 * self.urho + self.rho * s0)

    def step(self):
        self.moments()
        L = self.F
        tau = self.tau if self.nu is None else (self.phi * (self.nu[0] - self.nu[1]) + self.nu[1]) / L.cs2 + 0.5
        pre = 1 - 1 / (2 * tau)
        out = []
        for i, (c, w) in enumerate(zip(L.c, L.w)):
            cu = sum(k * u for k, u in zip(c, self.u) if k)
            cF = sum(k * F for k, F in zip(c, self.force) if k)
            cr = sum(k * g for k, g in zip(c, self.grad) if k)
            s = w * (cu / L.cs2 + cu * cu / (2 * L.cs2 ** 2) - self.uu / (2 * L.cs2))
            eq = self.p / L.cs2 * (w - (i == 0)) + self.rho * s
            src = pre * w * (cF / L.cs2 + cu * cr * (self.drho / L.cs2))
            out.append(self.f[i] - (self.f[i] - eq) / tau + src)
        now = sum(u * g for u, g in zip(self.u, self.grad))
        before = now if self.last is None else self.last
        drive = now if self.dgdt else 1.5 * now - 0.5 * before
        self.last = now
        gout = []
        for i, (c, w) in enumerate(zip(self.G.c, self.G.w)):
            c2 = sum(k * k for k in c)
            eq = w * self.alpha * self.mu if i else self.phi - (1 - w) * self.alpha * self.mu
            gout.append(eq + w * (-1 + (c2 - self.dim * self.G.cs2) / (2 * self.G.cs2)) * drive)   # tau_g = 1
        self.f = self.stream(L, out)
        self.g = self.stream(self.G, gout)

    def stream(self, L, star):
        """f_i(x) = f*_i(x - c_i); where x - c_i keeps none, the population that
        arrives from the other side, or the node's own when there is none."""
        new = [star[0]]
        for i in range(1, len(L.c)):
            o = L.opp[i]
            back = torch.where(self.known[o], _moved(star[o], L.c[o]), star[o])
            new.append(torch.where(self.known[i], _moved(star[i], L.c[i]), back))
        return [torch.where(self.zeta, v, 0.0) for v in new]

    def fields(self):
        self.moments()
        zero = torch.zeros_like(self.p)
        return (self.phi, torch.stack([torch.where(self.zeta, u, zero) for u in self.u], dim=-1),
                torch.where(self.zeta, self.p, zero))


def _solve64(lats, case):
    """(phi, u, p) after the case's steps, of lattices of one size and W, stacked."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    solid = torch.stack([torch.as_tensor(lat["solid"]) for lat in lats]).to(dev) != 0
    if lats[0]["field"] is not None:
        theta = torch.stack([torch.as_tensor(lat["field"]) for lat in lats]).double().to(dev)
    else:
        theta = torch.tensor([lat["theta"] for lat in lats], dtype=torch.float64, device=dev)
        theta = theta.reshape((-1,) + (1,) * (solid.dim() - 1))
    ref = _Reference(solid, theta, lats[0]["W"], case)
    ref.droplets(list(zip(*[lat["drops"] for lat in lats])))
    for _ in range(case["steps"]):
        ref.step()
    return (*ref.fields(), ref.zeta)


def exact(case, seed):
    if case["kind"] == "box":
        phi, u, p, _ = _solve64([_box(case, seed)], case)
        return {"phi": phi[0], "u": u[0], "p": p[0]}
    lats = _lattices(case, seed)
    groups = {}
    for k, lat in enumerate(lats):
        groups.setdefault((lat["solid"].shape, lat["W"]), []).append(k)
    parts = [None] * len(lats)
    for members in groups.values():
        phi, u, p, zeta = _solve64([lats[k] for k in members], case)
        for j, k in enumerate(members):
            parts[k] = (phi[j].reshape(-1), u[j].reshape(-1), p[j].reshape(-1))
    out = {name: torch.cat([part[q] for part in parts]) for q, name in enumerate(("phi", "u", "p"))}
    if case.get("angle"):
        out["mass"] = float(torch.where(zeta[0], phi[0], 0.0).sum())
        out["angle"] = None
    return out
