"""What the library's speed is measured on.

Every case goes through the public binding (``paper_2204_01117_gb300.uf``) as a
program that simulates wind around buildings calls it:

* ``steps``     time steps of one grid, then its fields (on the device);
* ``host``      fields up from pinned host memory, one step, fields down;
* ``channel``   the quasi-2D vortex street past a cylinder, fixed time step;
* ``batch``     many uneven grids advanced together;
* ``adjoint``   one design gradient: restart, forward steps, reverse sweep;
* ``design``    parametric design -> porosity and its vector-Jacobian product;
* ``mesh``      triangle meshes -> porosity;
* ``static``    the pressure solve that allocates no device memory.

``exact`` computes the same in 64 bits with plain torch: the time step from its
definition (staggered grid, MacCormack semi-Lagrangian advection with the Selle
clamp, explicit diffusion, porosity drag, projection, k-omega), the pressure by
diagonalising the operator along each axis.
"""
import math
import random

import numpy as np
import torch

from paper_2204_01117_gb300 import uf

FIELDS = ("u", "v", "w", "p", "k", "omega")
# what the vortex street is read from; its pressure after the impulsive start is only determined to about 1e-3 by the
# solver's residual tolerance (the channel is 768 cells long), whatever the solver
WAKE = ("u", "v", "w", "k", "omega")


def listed():
    return [
        # the smallest call: an interactive viewer steps once and reads the fields
        dict(name="view_48x40x16_f32", kind="steps", nx=48, ny=40, nz=16, precision="f32", wind=0.0, steps=1),
        # the double-precision validation run around one solid block (64 x 32 x 16)
        dict(name="block_64x32x16_f64", kind="steps", nx=64, ny=32, nz=16, precision="f64", wind=0.0, steps=10),
        # the ordinary production grid: a 512 m x 512 m urban block at 2 m
        dict(name="urban_256x256x64_f32", kind="steps", nx=256, ny=256, nz=64, precision="f32", wind=0.0, steps=4),
        # odd sizes and an oblique wind: two inflow and two outflow sides, ragged tiles on every axis
        dict(name="urban_157x203x41_f32", kind="steps", nx=157, ny=203, nz=41, precision="f32", wind=30.0, steps=4),
        # the largest: 33.5 M cells, far beyond the L2
        dict(name="urban_512x512x128_f32", kind="steps", nx=512, ny=512, nz=128, precision="f32", wind=0.0, steps=2),
        # double precision on an urban block, the reference run of a single-precision study
        dict(name="urban_128x96x40_f64", kind="steps", nx=128, ny=96, nz=40, precision="f64", wind=120.0, steps=2),
        # coupling with a host program: six fields up and down around every step
        dict(name="host_256x256x64_f32", kind="host", nx=256, ny=256, nz=64, precision="f32", wind=0.0),
        # the vortex-street validation, one cell thick
        dict(name="channel_512x768_f32", kind="channel", nx=512, ny=768, precision="f32", speed=5.0, steps=10),
        # a sweep over sites and wind directions advanced together
        dict(name="batch_8_f32", kind="batch", count=8, lo=96, hi=256, zlo=32, zhi=64, steps=2),
        # the step that a design gradient on the parametric lattice repeats: forward, taped, and reverse (over several steps
        # single precision decides by rounding on which side of a clamp it falls, and gradients cannot be compared)
        dict(name="adjoint_128x128x48_f32", kind="adjoint", nx=128, ny=128, nz=48, precision="f32", steps=1, ckpt=1),
        # the design map of that lattice and its transpose, every design iteration
        dict(name="design_128x128x48_f32", kind="design", nx=128, ny=128, nz=48, boxes=12),
        # a city of meshes to porosity, once per imported scene
        dict(name="mesh_256x256x64_f32", kind="mesh", nx=256, ny=256, nz=64, prisms=60, crowns=40, sub=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["steps", "steps", "steps", "f64", "channel", "batch", "adjoint", "design", "mesh", "static", "host"])
    if kind == "steps":
        return dict(kind="steps", nx=_log(rng, 40, 512), ny=_log(rng, 32, 512), nz=_log(rng, 9, 80), precision="f32",
                    wind=round(rng.uniform(0.0, 360.0), 1) if rng.random() < 0.6 else rng.choice([0.0, 90.0, 180.0, 270.0]),
                    steps=rng.randint(1, 3))
    if kind == "f64":
        return dict(kind="steps", nx=_log(rng, 40, 144), ny=_log(rng, 32, 144), nz=_log(rng, 9, 48), precision="f64",
                    wind=round(rng.uniform(0.0, 360.0), 1), steps=rng.randint(1, 3))
    if kind == "host":
        return dict(kind="host", nx=_log(rng, 48, 288), ny=_log(rng, 40, 256), nz=_log(rng, 12, 64), precision="f32",
                    wind=round(rng.uniform(0.0, 360.0), 1))
    if kind == "channel":
        return dict(kind="channel", nx=_log(rng, 256, 600), ny=_log(rng, 384, 900), precision="f32",
                    speed=round(rng.uniform(2.0, 20.0), 2), steps=rng.randint(4, 12))
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(3, 8), lo=rng.choice([48, 64, 96]), hi=rng.choice([128, 192, 224]), zlo=16,
                    zhi=56, steps=rng.randint(1, 3))
    if kind == "adjoint":
        return dict(kind="adjoint", nx=_log(rng, 48, 256), ny=_log(rng, 40, 192), nz=_log(rng, 16, 64), precision="f32", steps=1, ckpt=1)
    if kind == "design":
        return dict(kind="design", nx=_log(rng, 48, 192), ny=_log(rng, 40, 192), nz=_log(rng, 12, 48), boxes=rng.randint(1, 24))
    if kind == "mesh":
        return dict(kind="mesh", nx=_log(rng, 48, 256), ny=_log(rng, 40, 256), nz=_log(rng, 16, 64), prisms=rng.randint(4, 60),
                    crowns=rng.randint(2, 40), sub=rng.choice([2, 3, 4]))
    return dict(kind="static", nx=_log(rng, 40, 128), ny=_log(rng, 32, 112), nz=_log(rng, 8, 48), wind=round(rng.uniform(0.0, 360.0), 1))


# ------------------------------------------------------------------ inputs

def _params(case):
    """Grid parameters of a case (h = 2 m, log-law inflow, no-slip ground)."""
    kind = case["kind"]
    if kind == "channel":
        return dict(h=2e-3, wind_dir_deg=90.0, u_ref=case["speed"], inflow_loglaw=0, ground_noslip=0, fixed_dt=1e-4, I=1e-3, L=0.046)
    p = dict(h=2.0, wind_dir_deg=case.get("wind", 0.0), u_ref=3.0, z_ref=10.0, z0=0.5, inflow_loglaw=1, ground_noslip=1)
    if kind == "adjoint":
        p["fixed_dt"] = 0.2
    return p


def _overlap(lo, hi, n, h):
    """Fraction of each of the n cells of an axis inside [lo, hi]."""
    e = torch.arange(n + 1, dtype=torch.float64, device="cuda") * h
    return ((torch.clamp(e[1:], max=hi) - torch.clamp(e[:-1], min=lo)) / h).clamp(0.0, 1.0)


def _city_phi(nx, ny, nz, h, rng):
    """Porosity of a random urban block: solid boxes (footprint sides 10 to
    40 m, heights 10 to 60 m) as cut-cell volume fractions, and ellipsoidal
    canopies (porosity 0.3 to 0.8), 40 and 60 of them per 256 x 256 cells."""
    phi = torch.ones((nz, ny, nx), dtype=torch.float64, device="cuda")
    lx, ly, lz = nx * h, ny * h, nz * h
    area = nx * ny / 65536.0
    cells = lambda lo, hi, n: slice(max(0, int(lo / h)), min(n, int(hi / h) + 2))
    for _ in range(max(1, round(40 * area))):
        sx, sy = min(rng.uniform(10, 40), 0.3 * lx), min(rng.uniform(10, 40), 0.3 * ly)
        hz = min(rng.uniform(10, 60), 0.7 * lz)
        cx, cy = rng.uniform(0.1 * lx + sx / 2, 0.9 * lx - sx / 2), rng.uniform(0.1 * ly + sy / 2, 0.9 * ly - sy / 2)
        ox, oy, oz = _overlap(cx - sx / 2, cx + sx / 2, nx, h), _overlap(cy - sy / 2, cy + sy / 2, ny, h), _overlap(0.0, hz, nz, h)
        X, Y, Z = cells(cx - sx / 2, cx + sx / 2, nx), cells(cy - sy / 2, cy + sy / 2, ny), cells(0.0, hz, nz)
        v = phi[Z, Y, X]
        torch.minimum(v, 1.0 - oz[Z, None, None] * oy[None, Y, None] * ox[None, None, X], out=v)
    xs, ys, zs = ((torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) * h for n in (nx, ny, nz))
    for _ in range(max(1, round(60 * area))):
        r, ph, trunk = min(rng.uniform(3, 8), 0.2 * min(lx, ly)), rng.uniform(0.3, 0.8), rng.uniform(2, 5)
        cx, cy, cz = rng.uniform(0.1 * lx + r, 0.9 * lx - r), rng.uniform(0.1 * ly + r, 0.9 * ly - r), trunk + 0.75 * r
        X, Y, Z = cells(cx - r, cx + r, nx), cells(cy - r, cy + r, ny), cells(cz - 0.75 * r, cz + 0.75 * r, nz)
        d = ((xs[None, None, X] - cx) / r) ** 2 + ((ys[None, Y, None] - cy) / r) ** 2 + ((zs[Z, None, None] - cz) / (0.75 * r)) ** 2
        v = phi[Z, Y, X]
        torch.minimum(v, torch.where(d < 1.0, ph, 1.0), out=v)
    return phi


def _channel_phi(nx, ny, h, rng):
    """A solid cylinder of 0.046 m on a jittered axis, by cell centres."""
    xc, yc = nx * h / 2 + rng.uniform(-h, h), 0.4 * ny * h + rng.uniform(-h, h)
    x, y = ((torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) * h for n in (nx, ny))
    return ((x[None, :] - xc) ** 2 + (y[:, None] - yc) ** 2 > 0.023 ** 2).double()[None].contiguous()


def _lattice(nx, ny, h, count, rng):
    """Footprints of `count` square buildings of 20 m on an even lattice and
    their parameters (height, x shift, y shift)."""
    cols = max(1, int(math.ceil(math.sqrt(count * nx / ny))))
    rows = (count + cols - 1) // cols
    boxes, theta = [], []
    for q in range(count):
        cx, cy = nx * h * (q % cols + 1) / (cols + 1), ny * h * (q // cols + 1) / (rows + 1)
        boxes.append((cx - 10.0, cx + 10.0, cy - 10.0, cy + 10.0))
        theta.append((rng.uniform(20.0, 40.0), rng.uniform(-2.0, 2.0), rng.uniform(-2.0, 2.0)))
    return np.array(boxes), np.array(theta)


def _design_phi(nx, ny, nz, h, boxes, theta, width):
    """phi = prod (1 - chi) of the logistic boxes; theta may need a gradient."""
    x, y, z = ((torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) * h for n in (nx, ny, nz))
    phi = torch.ones((nz, ny, nx), dtype=torch.float64, device="cuda")
    s = torch.sigmoid
    for b, (H, dx, dy) in zip(boxes, theta):
        X = s((x - (b[0] + dx)) / width) * s(((b[1] + dx) - x) / width)
        Y = s((y - (b[2] + dy)) / width) * s(((b[3] + dy) - y) / width)
        phi = phi * (1.0 - s((H - z) / width)[:, None, None] * Y[None, :, None] * X[None, None, :])
    return phi


def _meshes(nx, ny, nz, h, prisms, crowns, rng):
    """Closed meshes: prism buildings (4 to 8 sides, radius 4 to 10 m) and
    canopies (subdivided octahedra projected onto ellipsoids)."""
    lx, ly, lz = nx * h, ny * h, nz * h
    tris, objects = [], []

    def add(t, ph):
        objects.append((sum(len(a) for a in tris), len(t), ph))
        tris.append(np.asarray(t, dtype=np.float64))

    for _ in range(prisms):
        cx, cy, r, n = rng.uniform(0.1 * lx, 0.9 * lx), rng.uniform(0.1 * ly, 0.9 * ly), rng.uniform(4.0, 10.0), rng.randint(4, 8)
        a0, H = rng.uniform(0.0, 6.28), rng.uniform(min(8.0, 0.5 * lz), 0.8 * lz)
        ring = [(cx + r * math.cos(a0 + 2 * math.pi * q / n), cy + r * math.sin(a0 + 2 * math.pi * q / n)) for q in range(n)]
        t = []
        for (x0, y0), (x1, y1) in zip(ring, ring[1:] + ring[:1]):
            t += [[(cx, cy, 0.0), (x1, y1, 0.0), (x0, y0, 0.0)], [(cx, cy, H), (x0, y0, H), (x1, y1, H)],
                  [(x0, y0, 0.0), (x1, y1, 0.0), (x1, y1, H)], [(x0, y0, 0.0), (x1, y1, H), (x0, y0, H)]]
        add(t, 0.0)
    for _ in range(crowns):
        c = np.array([rng.uniform(0.1 * lx, 0.9 * lx), rng.uniform(0.1 * ly, 0.9 * ly), rng.uniform(4.0, 10.0)])
        r = rng.uniform(3.0, 6.0)
        t = [[(sx, 0, 0), (0, sy, 0), (0, 0, sz)] for sx in (1, -1) for sy in (1, -1) for sz in (1, -1)]
        t = np.array(t, dtype=np.float64)
        for _ in range(2):
            a, b, d = t[:, 0], t[:, 1], t[:, 2]
            ab, bd, da = a + b, b + d, d + a
            t = np.concatenate([np.stack(q, 1) for q in ((a, ab, da), (b, bd, ab), (d, da, bd), (ab, bd, da))])
            t = t / np.linalg.norm(t, axis=2, keepdims=True)
        add(t * r * np.array([1.0, 1.0, 0.75]) + c, rng.uniform(0.3, 0.8))
    return np.concatenate(tris), objects


def _instances(case, rng):
    out = []
    for _ in range(case["count"]):
        nx, ny = (16 * rng.randint(case["lo"] // 16, case["hi"] // 16) for _ in range(2))
        nz = 8 * rng.randint(case["zlo"] // 8, case["zhi"] // 8)
        out.append(dict(nx=nx, ny=ny, nz=nz, h=2.0, wind_dir_deg=rng.uniform(0.0, 360.0), u_ref=rng.uniform(2.0, 8.0), z_ref=10.0,
                        z0=0.5, inflow_loglaw=1, ground_noslip=1))
    return out


def _batch_shape(case):
    """The instances' sizes belong to the case; wind, speed and city to the seed."""
    return random.Random(case["count"] * 1000003 + case["lo"] * 1009 + case["hi"] * 31 + case["zhi"])


def _batch_inputs(case, seed):
    insts, r = _instances(case, _batch_shape(case)), random.Random(seed)
    return insts, [_city_phi(p["nx"], p["ny"], p["nz"], p["h"], r) for p in insts]


def _static_b(case, seed):
    """A right-hand side as a step forms it: sources and sinks at the faces of obstacles, on a smooth background."""
    r = random.Random(seed)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    phi = _city_phi(nx, ny, nz, 2.0, r)
    b = torch.zeros_like(phi)
    b[:, :, 1:] = phi[:, :, 1:] - phi[:, :, :-1]
    g = torch.Generator(device="cuda").manual_seed(seed)
    return (10.0 * b + 0.01 * torch.randn(phi.shape, generator=g, device="cuda", dtype=torch.float64)).float()


def _case_phi(case, seed):
    r, nx, ny = random.Random(seed), case["nx"], case["ny"]
    if case["kind"] == "channel":
        return _channel_phi(nx, ny, 2e-3, r)
    if case["kind"] == "adjoint":
        boxes, theta = _lattice(nx, ny, 2.0, 12 if nx * ny >= 96 * 96 else 4, r)
        return _design_phi(nx, ny, case["nz"], 2.0, boxes, theta, 2.0)
    return _city_phi(nx, ny, case["nz"], 2.0, r)


def _checkpoint(case, phi):
    """Fields three steps into the flow, computed in 64 bits and rounded."""
    s = _Step(case["nx"], case["ny"], case["nz"], phi.double(), **_params(case))
    for _ in range(3):
        s.step()
    return {n: f.float().contiguous() for n, f in s.fields().items()}


def _cast(phi, precision):
    return phi if precision == "f64" else phi.float()


def _buffers(g, device, names=FIELDS):
    if device == "cuda":
        return {n: torch.empty(g.shapes[n], dtype=g.torch_dtype, device="cuda") for n in names}
    return {n: torch.empty(g.shapes[n], dtype=g.torch_dtype, pin_memory=True) for n in names}


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("steps", "channel", "host", "adjoint"):
        g = uf.Grid(case["nx"], case["ny"], case.get("nz", 1), precision=case["precision"], **_params(case))
        phi = _cast(_case_phi(case, seed), case["precision"])
        g.set_porosity(phi)
        if kind == "adjoint":   # the state a checkpoint holds: some steps into the flow
            return dict(case=case, grid=g, x0=_checkpoint(case, phi), dphi=torch.empty(g.shapes["phi"], dtype=g.torch_dtype, device="cuda"))
        g.init_state()
        s = dict(case=case, grid=g, out=_buffers(g, "cuda", WAKE if kind == "channel" else FIELDS))
        if kind == "host":
            s["host"], s["out"] = g.take_fields(_buffers(g, "host")), _buffers(g, "host")
        return s
    if kind == "batch":
        insts, phis = _batch_inputs(case, seed)
        b = uf.Batch(insts)
        for g, phi in zip(b.grids, phis):
            g.set_porosity(phi.float())
            g.init_state()
        return dict(case=case, batch=b, out=[_buffers(g, "cuda") for g in b.grids])
    if kind == "design":
        g = uf.Grid(case["nx"], case["ny"], case["nz"], **_params(case))
        boxes, theta = _lattice(case["nx"], case["ny"], 2.0, case["boxes"], random.Random(seed))
        return dict(case=case, grid=g, boxes=boxes, theta=theta, phi=torch.empty(g.shapes["phi"], device="cuda"),
                    lam=torch.randn(g.shapes["phi"], generator=torch.Generator(device="cuda").manual_seed(seed), device="cuda"))
    if kind == "mesh":
        g = uf.Grid(case["nx"], case["ny"], case["nz"], **_params(case))
        tris, objects = _meshes(case["nx"], case["ny"], case["nz"], 2.0, case["prisms"], case["crowns"], random.Random(seed))
        return dict(case=case, grid=g, tris=tris, objects=objects, phi=torch.empty(g.shapes["phi"], device="cuda"))
    b = _static_b(case, seed)
    return dict(case=case, b=b, stream=torch.cuda.Stream())


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind in ("steps", "channel"):
        s["grid"].run(case["steps"], stats=False)
        return s["grid"].take_fields(s["out"])
    if kind == "host":
        s["grid"].put_fields(s["host"])
        s["grid"].step(stats=False)
        return s["grid"].take_fields(s["out"])
    if kind == "batch":
        s["batch"].run(case["steps"], stats=False)
        return [g.take_fields(o) for g, o in zip(s["batch"].grids, s["out"])]
    if kind == "adjoint":
        s["grid"].put_fields(s["x0"])
        J, g = s["grid"].adjoint_run(case["steps"], case["ckpt"], out=s["dphi"])
        return {"J": J, "dphi": g}
    if kind == "design":
        phi = s["grid"].design_to_phi(s["boxes"], s["theta"], 2.0, out=s["phi"])
        return {"phi": phi, "grad": s["grid"].design_vjp(s["boxes"], s["theta"], 2.0, s["lam"])}
    if kind == "mesh":
        return s["grid"].mesh_to_phi(s["tris"], s["objects"], case["sub"], out=s["phi"])
    p = torch.zeros_like(s["b"])
    s["stream"].wait_stream(torch.cuda.current_stream())
    uf.poisson_solve_static(s["b"], p, case["wind"], stream=s["stream"])
    return p


# -------------------------------------------------------------------- work

def work(case):
    """Bytes: each step reads u, v, w, p, k, omega and the porosity and writes
    the six fields; the reverse sweep does so twice over.  Flops: about 900 a
    cell and step without the pressure solve, and 300 for one."""
    kind = case["kind"]
    size = 8 if case.get("precision") == "f64" else 4
    if kind == "batch":
        n = sum(p["nx"] * p["ny"] * p["nz"] for p in _instances(case, _batch_shape(case)))
    else:
        n = case["nx"] * case["ny"] * case.get("nz", 1)
    if kind in ("steps", "channel", "batch"):
        return {"bytes": 13.0 * size * n * case["steps"], "flops": 1200.0 * n * case["steps"]}
    if kind == "host":
        return {"bytes": (13.0 + 12.0) * size * n, "flops": 1200.0 * n}
    if kind == "adjoint":
        return {"bytes": 39.0 * size * n * case["steps"], "flops": 4000.0 * n * case["steps"]}
    if kind == "design":
        return {"bytes": 8.0 * n, "flops": 20.0 * n * case["boxes"]}
    if kind == "mesh":
        return {"bytes": 4.0 * n + 72.0 * (24 * case["prisms"] + 128 * case["crowns"]),
                "flops": 40.0 * case["sub"] ** 3 * (24 * 1500.0 * case["prisms"] + 128 * 100.0 * case["crowns"])}
    return {"bytes": 8.0 * n, "flops": 300.0 * n}


# -------------------------------------------------- the same in 64 bits ----

INFLOW, OUTFLOW, SLIP, NOSLIP = range(4)


class _Step:
    """The time step in 64 bits on (z, y, x) tensors."""

    def __init__(self, nx, ny, nz, phi, h, wind_dir_deg, u_ref, inflow_loglaw, ground_noslip, z_ref=10.0, z0=0.5, fixed_dt=0.0, I=0.1,
                 L=10.0):
        self.n, self.h, self.fixed_dt = (nx, ny, nz), h, fixed_dt
        self.rho, self.nu, self.C_mu, self.C_lim = 1.225, 1.5e-5, 0.09, 7.0 / 8.0
        th = math.radians(wind_dir_deg)
        self.dir = (math.cos(th), math.sin(th))
        side = lambda c: INFLOW if c > 1e-9 else OUTFLOW if c < -1e-9 else SLIP
        self.side = [side(self.dir[0]), side(-self.dir[0]), side(self.dir[1]), side(-self.dir[1]), NOSLIP if ground_noslip else SLIP, SLIP]
        z = (torch.arange(nz, dtype=torch.float64, device="cuda") + 0.5) * h
        self.prof = torch.clamp(u_ref * torch.log(z / z0) / math.log(z_ref / z0), min=0.0) if inflow_loglaw else torch.full_like(z, u_ref)
        uin = u_ref
        self.k_in = 1.5 * (I * uin) ** 2
        self.om_in = math.sqrt(self.k_in) / (self.C_mu ** 0.25 * L)
        self.c = 1.0 * 0.62 * torch.clamp((1.0 - phi) / (phi + 1e-10), min=0.0) ** 2.5
        self.modes = [self._modes(m, a) for a, m in enumerate(self.n)]
        col = self.prof[:, None, None]
        self.u = (col * self.dir[0]).expand(nz, ny, nx + 1).clone()
        self.v = (col * self.dir[1]).expand(nz, ny + 1, nx).clone()
        self.w = torch.zeros((nz + 1, ny, nx), dtype=torch.float64, device="cuda")
        self.k = torch.full((nz, ny, nx), self.k_in, dtype=torch.float64, device="cuda")
        self.om = torch.full((nz, ny, nx), self.om_in, dtype=torch.float64, device="cuda")
        self._bc(self.u, self.v, self.w)
        dt = self._dt()
        self._drag(dt, self.u, self.v, self.w)
        self._project(dt)

    def _modes(self, m, axis):
        T = torch.zeros((m, m), dtype=torch.float64, device="cuda")
        d = torch.full((m,), 2.0, dtype=torch.float64, device="cuda")
        d[0] -= 0.0 if self.side[2 * axis] == OUTFLOW else 1.0
        d[-1] -= 0.0 if self.side[2 * axis + 1] == OUTFLOW else 1.0
        T.diagonal().copy_(d)
        if m > 1:
            T.diagonal(1).fill_(-1.0)
            T.diagonal(-1).fill_(-1.0)
        return torch.linalg.eigh(T)

    def solve(self, b):
        (lx, X), (ly, Y), (lz, Z) = self.modes
        t = torch.einsum("kc,cji->kji", Z.T, torch.einsum("jc,kci->kji", Y.T, b @ X))
        t /= lz[:, None, None] + ly[None, :, None] + lx[None, None, :]
        return torch.einsum("kc,cji->kji", Z, torch.einsum("jc,kci->kji", Y, t @ X.T))

    def _dt(self):
        return self.fixed_dt if self.fixed_dt > 0 else 0.5 * self.h / float(max(self.u.abs().max(), self.v.abs().max(), self.w.abs().max()))

    def _bc(self, u, v, w):
        col = self.prof[:, None]
        val = lambda s, inner, inflow: inflow.expand_as(inner) if s == INFLOW else inner if s == OUTFLOW else torch.zeros_like(inner)
        u[:, :, 0], u[:, :, -1] = val(self.side[0], u[:, :, 1].clone(), col * self.dir[0]), val(self.side[1], u[:, :, -2].clone(), col * self.dir[0])
        v[:, 0], v[:, -1] = val(self.side[2], v[:, 1].clone(), col * self.dir[1]), val(self.side[3], v[:, -2].clone(), col * self.dir[1])
        w[0], w[-1] = 0.0, 0.0

    def _strain2(self):
        u, v, w, ih = self.u, self.v, self.w, 1.0 / self.h
        uc, vc, wc = 0.5 * (u[:, :, 1:] + u[:, :, :-1]), 0.5 * (v[:, 1:] + v[:, :-1]), 0.5 * (w[1:] + w[:-1])

        def grad(f, dim):
            m = f.shape[dim]
            i = torch.arange(m, device="cuda")
            p, q = (i + 1).clamp(max=m - 1), (i - 1).clamp(min=0)
            shape = [1, 1, 1]
            shape[dim] = m
            s = torch.where(p > q, ih / (p - q).clamp(min=1).double(), torch.zeros((), dtype=torch.float64, device="cuda")).view(shape)
            return (f.index_select(dim, p) - f.index_select(dim, q)) * s

        sxx, syy, szz = (u[:, :, 1:] - u[:, :, :-1]) * ih, (v[:, 1:] - v[:, :-1]) * ih, (w[1:] - w[:-1]) * ih
        sxy, sxz, syz = 0.5 * (grad(uc, 1) + grad(vc, 2)), 0.5 * (grad(uc, 0) + grad(wc, 2)), 0.5 * (grad(vc, 0) + grad(wc, 1))
        return sxx ** 2 + syy ** 2 + szz ** 2 + 2.0 * (sxy ** 2 + sxz ** 2 + syz ** 2)

    def _nut(self, S2, dt):
        om = torch.maximum(self.om, self.C_lim * torch.sqrt(S2) / math.sqrt(self.C_mu * 0.5))
        return torch.clamp(torch.clamp(self.k / om, max=self.h * self.h / (6.0 * dt) - self.nu), min=0.0)

    @staticmethod
    def _axis(m, off, dim):
        """Lower cell, upper cell and weight of lattice index + off along an axis of m points."""
        shape = [1, 1, 1]
        shape[dim] = -1
        lo = torch.floor(off)
        f = torch.arange(off.shape[dim], device="cuda").view(shape) + lo.long()
        t = off - lo
        t = torch.where(f < 0, 0.0, t)
        t = torch.where(f >= m - 1, 1.0 if m >= 2 else 0.0, t)
        f = f.clamp(0, max(m - 2, 0))
        return f, (f + 1).clamp(max=m - 1), t

    def _sample(self, F, ox, oy, oz, spread=False):
        """F at (own lattice index + offsets); the offsets are tensors of the sampled points' shape."""
        Lz, Ly, Lx = F.shape
        (x0, x1, tx), (y0, y1, ty), (z0, z1, tz) = self._axis(Lx, ox, 2), self._axis(Ly, oy, 1), self._axis(Lz, oz, 0)
        flat, mn, mx, planes = F.reshape(-1), None, None, []
        for z in (z0, z1):
            rows = []
            for y in (y0, y1):
                base = (z * Ly + y) * Lx
                a, b = flat[base + x0], flat[base + x1]
                if spread:
                    lo, hi = torch.minimum(a, b), torch.maximum(a, b)
                    mn, mx = (lo, hi) if mn is None else (torch.minimum(mn, lo), torch.maximum(mx, hi))
                rows.append(a + tx * (b - a))
            planes.append(rows[0] + ty * (rows[1] - rows[0]))
        r = planes[0] + tz * (planes[1] - planes[0])
        return (r, mn, mx) if spread else r

    def _advect(self, dt):
        s, F, out = dt / self.h, (self.u, self.v, self.w), []
        for q in range(3):
            full = lambda c, q=q: torch.full(F[q].shape, c, dtype=torch.float64, device="cuda")
            d = []
            for r in range(3):
                if r == q:
                    d.append(s * F[q])
                    continue
                # the lattices of q and r are half a cell apart along both axes
                off = [0.0, 0.0, 0.0]
                off[q], off[r] = -0.5, 0.5
                d.append(s * self._sample(F[r], full(off[0]), full(off[1]), full(off[2])))
            fwd, mn, mx = self._sample(F[q], -d[0], -d[1], -d[2], spread=True)
            bwd = self._sample(fwd, d[0], d[1], d[2])
            out.append(torch.minimum(torch.maximum(fwd + 0.5 * (F[q] - bwd), mn), mx))
            del fwd, bwd, mn, mx, d
        return out

    def _ghosts(self, f, dim, lo, hi, inflow):
        """f with one ghost plane on each side along dim (tangential rule)."""
        m = f.shape[dim]

        def ghost(s, q):
            return inflow.expand_as(q) if s == INFLOW else -q if s == NOSLIP else q

        return torch.cat([ghost(lo, f.narrow(dim, 0, 1)), f, ghost(hi, f.narrow(dim, m - 1, 1))], dim)

    def _diffuse(self, dt, nut, u, v, w):
        self._bc(u, v, w)
        c, S = dt / (self.h * self.h), self.side
        zero = torch.zeros((1, 1, 1), dtype=torch.float64, device="cuda")
        new = []
        for q, f in enumerate((u, v, w)):
            ax = 2 - q
            inflow = zero if q == 2 else self.prof[:, None, None] * self.dir[q]
            lap = -6.0 * f
            for a in range(3):   # axis a: x, y, z
                dim = 2 - a
                if a == q:
                    e = torch.cat([f.narrow(dim, 0, 1), f, f.narrow(dim, f.shape[dim] - 1, 1)], dim)   # boundary faces are not kept
                else:
                    e = self._ghosts(f, dim, S[2 * a], S[2 * a + 1], inflow if a != 2 else zero)
                lap += e.narrow(dim, 0, f.shape[dim]) + e.narrow(dim, 2, f.shape[dim])
            m = f.shape[ax]
            r = f.clone()
            r.narrow(ax, 1, m - 2).add_(c * (self.nu + 0.5 * (nut.narrow(ax, 0, m - 2) + nut.narrow(ax, 1, m - 2))) * lap.narrow(ax, 1, m - 2))
            new.append(r)
        self._bc(*new)
        return new

    def _drag(self, dt, u, v, w):
        """Drag on the interior faces from fields with their boundary values, then the boundary values of the result."""
        f, c, new = (u, v, w), self.c, []
        for q in range(3):
            ax = 2 - q
            m = f[q].shape[ax]
            own = f[q].narrow(ax, 1, m - 2)
            sq = own * own
            for r in range(3):
                if r == q:
                    continue
                rx = 2 - r
                a = f[r].narrow(rx, 0, f[r].shape[rx] - 1) + f[r].narrow(rx, 1, f[r].shape[rx] - 1)   # on cells
                a = 0.25 * (a.narrow(ax, 0, m - 2) + a.narrow(ax, 1, m - 2))
                sq = sq + a * a
            cf = 0.5 * (c.narrow(ax, 0, m - 2) + c.narrow(ax, 1, m - 2))
            n = f[q].clone()
            n.narrow(ax, 1, m - 2).mul_(torch.clamp(1.0 - dt * cf * torch.sqrt(sq), min=0.0))
            new.append(n)
        self._bc(*new)
        self.u, self.v, self.w = new

    def _project(self, dt):
        u, v, w = self.u, self.v, self.w
        div = (u[:, :, 1:] - u[:, :, :-1]) + (v[:, 1:] - v[:, :-1]) + (w[1:] - w[:-1])
        self.p = p = self.solve(-(self.rho * self.h / dt) * div)
        g = dt / (self.rho * self.h)
        u[:, :, 1:-1] -= g * (p[:, :, 1:] - p[:, :, :-1])
        v[:, 1:-1] -= g * (p[:, 1:] - p[:, :-1])
        w[1:-1] -= g * (p[1:] - p[:-1])
        if self.side[0] == OUTFLOW:
            u[:, :, 0] -= g * p[:, :, 0]
        if self.side[1] == OUTFLOW:
            u[:, :, -1] += g * p[:, :, -1]
        if self.side[2] == OUTFLOW:
            v[:, 0] -= g * p[:, 0]
        if self.side[3] == OUTFLOW:
            v[:, -1] += g * p[:, -1]

    def _turbulence(self, dt):
        u, v, w, k, om, ih = self.u, self.v, self.w, self.k, self.om, 1.0 / self.h
        S2 = self._strain2()
        nut = self._nut(S2, dt)
        vel = (0.5 * (u[:, :, 1:] + u[:, :, :-1]), 0.5 * (v[:, 1:] + v[:, :-1]), 0.5 * (w[1:] + w[:-1]))
        rates = []
        for f, fin in ((k, self.k_in), (om, self.om_in)):
            adv, lap = torch.zeros_like(f), -6.0 * f
            for a in range(3):
                dim = 2 - a
                m = f.shape[dim]
                end = lambda s, q: torch.full_like(q, fin) if s == INFLOW else q
                e = torch.cat([end(self.side[2 * a], f.narrow(dim, 0, 1)), f, end(self.side[2 * a + 1], f.narrow(dim, m - 1, 1))], dim)
                lo, hi = e.narrow(dim, 0, m), e.narrow(dim, 2, m)
                lap = lap + lo + hi
                adv = adv + vel[a] * torch.where(vel[a] > 0, f - lo, hi - f) * ih
            rates.append((adv, lap * ih * ih))
        rk = -rates[0][0] + 2.0 * nut * S2 - self.C_mu * k * om + (self.nu + 0.6 * nut) * rates[0][1]
        ro = -rates[1][0] + 2.0 * 0.52 * S2 - 0.0708 * om * om + (self.nu + 0.5 * nut) * rates[1][1]
        self.k, self.om = torch.clamp(k + dt * rk, min=1e-10), torch.clamp(om + dt * ro, min=1e-6)

    def step(self):
        dt = self._dt()
        nut = self._nut(self._strain2(), dt)
        self._drag(dt, *self._diffuse(dt, nut, *self._advect(dt)))
        self._project(dt)
        self._turbulence(dt)

    def fields(self):
        return {"u": self.u, "v": self.v, "w": self.w, "p": self.p, "k": self.k, "omega": self.om}

    def comfort(self, z_lo=1.0, z_hi=3.0, u_hi=4.0, u_lo=1.0):
        z = (torch.arange(self.n[2], dtype=torch.float64, device="cuda") + 0.5) * self.h
        on = ((z >= z_lo - 1e-9) & (z <= z_hi + 1e-9))[:, None, None]
        u, v, w = self.u, self.v, self.w
        s = torch.sqrt((0.5 * (u[:, :, 1:] + u[:, :, :-1])) ** 2 + (0.5 * (v[:, 1:] + v[:, :-1])) ** 2 + (0.5 * (w[1:] + w[:-1])) ** 2)
        return float((((s - u_hi).clamp(min=0.0) ** 2 + (u_lo - s).clamp(min=0.0) ** 2) * on).sum())


def _mesh_phi(case, tris, objects):
    """Even-odd ray casting, every operation rounded on its own (a torch operation each)."""
    nx, ny, nz, sub, h = case["nx"], case["ny"], case["nz"], case["sub"], 2.0
    off = (torch.arange(sub, dtype=torch.float64, device="cuda") + 0.5) / sub
    vals = torch.ones((nz, ny, nx, sub ** 3), dtype=torch.float64, device="cuda")
    rx, ry, rz = 0.5741, 0.6219, 0.5327
    dot = lambda a, b: (a[0] * b[0] + a[1] * b[1]) + a[2] * b[2]
    for first, count, ph in objects:
        t = tris[first:first + count]
        lo, hi = t.reshape(-1, 3).min(0), t.reshape(-1, 3).max(0)
        rng = [(max(0, int(lo[a] / h) - 1), min(m, int(hi[a] / h) + 2)) for a, m in enumerate((nx, ny, nz))]
        if any(a >= b for a, b in rng):
            continue
        ax = [(torch.arange(a, b, dtype=torch.float64, device="cuda")[:, None] + off) * h for a, b in rng]
        shape = tuple(b - a for a, b in reversed(rng))
        px = ax[0].view(1, 1, shape[2], 1, 1, sub).expand(*shape, sub, sub, sub).reshape(*shape, -1)
        py = ax[1].view(1, shape[1], 1, 1, sub, 1).expand(*shape, sub, sub, sub).reshape(*shape, -1)
        pz = ax[2].view(shape[0], 1, 1, sub, 1, 1).expand(*shape, sub, sub, sub).reshape(*shape, -1)
        n = torch.zeros(px.shape, dtype=torch.int32, device="cuda")
        for v in t:
            e1, e2 = [float(v[1][a]) - float(v[0][a]) for a in range(3)], [float(v[2][a]) - float(v[0][a]) for a in range(3)]
            q = (ry * e2[2] - rz * e2[1], rz * e2[0] - rx * e2[2], rx * e2[1] - ry * e2[0])
            det = dot(e1, q)
            if det == 0.0:
                continue
            s, adet = (1.0, det) if det > 0 else (-1.0, -det)
            T = (px - float(v[0][0]), py - float(v[0][1]), pz - float(v[0][2]))
            u = dot(T, q) * s
            r = (T[1] * e1[2] - T[2] * e1[1], T[2] * e1[0] - T[0] * e1[2], T[0] * e1[1] - T[1] * e1[0])
            w, d = dot((rx, ry, rz), r) * s, dot(e2, r) * s
            n += ((u >= 0) & (u <= adet) & (w >= 0) & (u + w <= adet) & (d > 0)).int()
        inside = (n & 1).bool() & (px >= lo[0]) & (px <= hi[0]) & (py >= lo[1]) & (py <= hi[1]) & (pz >= lo[2]) & (pz <= hi[2])
        view = vals[rng[2][0]:rng[2][1], rng[1][0]:rng[1][1], rng[0][0]:rng[0][1]]
        view.copy_(torch.where(inside, view.clamp(max=ph), view))
    return vals.mean(-1)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("steps", "channel", "host", "adjoint"):
        phi = _cast(_case_phi(case, seed), case["precision"]).double()
        s = _Step(case["nx"], case["ny"], case.get("nz", 1), phi, **_params(case))
        if kind == "adjoint":
            x = {n: f.double() for n, f in _checkpoint(case, phi).items()}
            s.u, s.v, s.w, s.k, s.om = x["u"], x["v"], x["w"], x["k"], x["omega"]
        for _ in range(1 if kind == "host" else case["steps"]):
            s.step()
        if kind == "adjoint":   # the gradient is one-sided at the clamps' ties, where 64 bits decide otherwise: no value for it
            return {"J": s.comfort(), "dphi": None}
        return {n: f for n, f in s.fields().items() if kind != "channel" or n in WAKE}
    if kind == "batch":
        out = []
        for p, phi in zip(*_batch_inputs(case, seed)):
            s = _Step(phi=phi.float().double(), **p)
            for _ in range(case["steps"]):
                s.step()
            out.append(s.fields())
        return out
    if kind == "design":
        boxes, theta = _lattice(case["nx"], case["ny"], 2.0, case["boxes"], random.Random(seed))
        th = torch.tensor(theta, device="cuda", requires_grad=True)
        phi = _design_phi(case["nx"], case["ny"], case["nz"], 2.0, torch.tensor(boxes, device="cuda"), th, 2.0)
        lam = torch.randn(phi.shape, generator=torch.Generator(device="cuda").manual_seed(seed), device="cuda").double()
        (g,) = torch.autograd.grad((phi * lam).sum(), th)
        return {"phi": phi.detach(), "grad": g.reshape(-1)}
    if kind == "mesh":
        return _mesh_phi(case, *_meshes(case["nx"], case["ny"], case["nz"], 2.0, case["prisms"], case["crowns"], random.Random(seed)))
    b = _static_b(case, seed).double()
    s = _Step(case["nx"], case["ny"], case["nz"], torch.ones_like(b), h=2.0, wind_dir_deg=case["wind"], u_ref=1.0, inflow_loglaw=0, ground_noslip=0)
    return s.solve(b)
