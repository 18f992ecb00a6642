"""Workloads of the FLIP step library: what a program that uses it has it do.

A simulation program owns the particles of a scene, hands them to the library, advances one
displayed frame (1/60 s = 4 steps of the default dt = 1/240) and takes the particles and the grid
fields back; a caller with its own grid asks for the pressure solve alone; a renderer asks for the
scalar field of the particles and for the mesh of a level set.  Each case below is one such call
through paper_2404_01931_gb300.flip, on the scenes (dam break, double dam break, water drop, drop
into pool) and grids (32^3 .. 256^3) of this project's tests and benchmark.

Cases are stationary: every pass starts from the same particles, so it can be repeated.  Particles
come back in creation order, since the order inside a cell is not specified.
"""
import math

import numpy as np
import torch

from paper_2404_01931_gb300 import flip as F

DT = 1.0 / 240.0
GRAVITY = -9.81
FLIP_RATIO = 0.95
STEPS = 4
FIELDS = (F.U_NEW, F.V_NEW, F.W_NEW, F.PRESSURE)

# Scene geometry in units of the longest edge (x < a, y < b, ...), as in scenes.py.
#   dam     block at the x = 0 wall, quarter width and half height
#   ddam    two blocks at the x walls
#   drop    a free sphere falling to the floor
#   pool    a pool and a sphere falling into it
#   wide    a square-root block (x < a, y < a) of the batched scenes, a given by "frac"


def listed():
    return [
        # The smallest grid of the paper's tables: launches, barriers and latency count.
        dict(name="dam32_fp32", kind="frame", scene="dam", nx=32, ny=32, nz=32, precision="fp32",
             frac=0.0, warm=False, grid_advect=False),
        # The middle grid of those tables, to the tight tolerance.
        dict(name="ddam64_mixed", kind="frame", scene="ddam", nx=64, ny=64, nz=64,
             precision="mixed", frac=0.0, warm=False, grid_advect=False),
        # The largest grid of those tables at the library's default precision.
        dict(name="dam128_fp32", kind="frame", scene="dam", nx=128, ny=128, nz=128,
             precision="fp32", frac=0.0, warm=False, grid_advect=False),
        # A production scene of a few million particles on the same grid, tight tolerance.
        dict(name="pool128_mixed", kind="frame", scene="pool", nx=128, ny=128, nz=128,
             precision="mixed", frac=0.0, warm=False, grid_advect=False),
        # The benchmark's workload: 42 M particles.
        dict(name="pool256_mixed", kind="frame", scene="pool", nx=256, ny=256, nz=256,
             precision="mixed", frac=0.0, warm=False, grid_advect=False),
        # An odd box: no extent a multiple of a brick, particles moved by the grid velocity.
        dict(name="ragged_gridadv", kind="frame", scene="pool", nx=101, ny=67, nz=83,
             precision="mixed", frac=0.0, warm=False, grid_advect=True),
        # A scene submitted whole: created, advanced a frame with the adaptive time step and
        # reseeding to 3..12 particles per cell (Sec. 3.1.2, 3.1.4), read, destroyed.
        dict(name="oneshot_reseed64", kind="oneshot", scene="ddam", nx=64, ny=64, nz=64,
             precision="fp32", frac=0.0),
        # Many small scenes advanced together, as a simulation service does.
        dict(name="batch16", kind="batch", count=16, lo=32, hi=96, precision="mixed", shape_seed=0),
        # The pressure solve alone, for a caller with its own grid.
        dict(name="solve72", kind="solve", nx=72, ny=64, nz=80),
        # A frame's scalar field for the surface at two sizes.
        dict(name="sdf128", kind="sdf", scene="dam", nx=128, ny=128, nz=128, frac=0.0),
        dict(name="sdf256", kind="sdf", scene="pool", nx=256, ny=256, nz=256, frac=0.0),
        # Its mesh: marching cubes and vertex normals of a level set.
        dict(name="mesh160", kind="mesh", nx=160, ny=160, nz=160, radius=0.31),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["frame", "frame", "frame", "frame", "oneshot", "batch", "solve", "sdf",
                       "mesh"])
    if kind in ("frame", "sdf", "oneshot"):
        n = _log_int(rng, 24, {"frame": 240, "sdf": 200, "oneshot": 80}[kind])
        dims = [n, n, n]
        if rng.random() < 0.6:  # a ragged box: two extents below the first
            dims[1] = max(16, int(n * rng.uniform(0.55, 1.0)))
            dims[2] = max(16, int(n * rng.uniform(0.55, 1.0)))
        scene = rng.choice(["dam", "ddam", "drop", "pool", "wide"])
        case = dict(kind=kind, scene=scene, nx=dims[0], ny=dims[1], nz=dims[2],
                    frac=round(rng.uniform(0.45, 0.65), 4) if scene == "wide" else 0.0)
        if kind != "sdf":
            case["precision"] = rng.choice(["fp32", "mixed"])
        if kind == "frame":
            case["warm"] = case["precision"] == "mixed" and rng.random() < 0.2
            case["grid_advect"] = rng.random() < 0.2
        return case
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(2, 16), lo=24, hi=rng.randint(40, 96),
                    precision=rng.choice(["fp32", "mixed"]), shape_seed=rng.randrange(1 << 20))
    if kind == "solve":
        return dict(kind="solve", nx=_log_int(rng, 16, 100), ny=_log_int(rng, 16, 100),
                    nz=_log_int(rng, 16, 100))
    return dict(kind="mesh", nx=_log_int(rng, 24, 220), ny=_log_int(rng, 24, 220),
                nz=_log_int(rng, 24, 220), radius=round(rng.uniform(0.2, 0.4), 4))


# ------------------------------------------------------------------ geometry

def _fluid_mask(case, device):
    """bool[nz, ny, nx]: the cells seeded with particles."""
    n = (case["nx"], case["ny"], case["nz"])
    big = max(n)
    dx = 1.0 / big
    ext = [a * dx for a in n]
    x, y, z = (((torch.arange(a, device=device, dtype=torch.float64) + 0.5) * dx) for a in n)
    x, y, z = x[None, None, :], y[None, :, None], z[:, None, None]
    s = case["scene"]
    if s == "dam":
        m = (x < 0.25 * ext[0]) & (y < 0.5 * ext[1]) & (z > -1.0)
    elif s == "ddam":
        m = ((x < 0.2 * ext[0]) | (x > 0.8 * ext[0])) & (y < 0.5 * ext[1]) & (z > -1.0)
    elif s == "wide":
        m = (x < case["frac"] * ext[0]) & (y < case["frac"] * ext[1]) & (z > -1.0)
    else:
        r, cy = (0.2, 0.6) if s == "drop" else (0.15, 0.7)
        r *= min(ext)
        m = ((x - 0.5 * ext[0]) ** 2 + (y - cy * ext[1]) ** 2 + (z - 0.5 * ext[2]) ** 2) < r * r
        if s == "pool":
            m = m | ((y < 0.3 * ext[1]) & (x > -1.0) & (z > -1.0))
    return m


def _particles(case, seed, device="cuda"):
    """Six float32 arrays: 8 particles per fluid cell (jittered 2x2x2 sub-cells), moving with a
    smooth divergence-free velocity of random phases, a falling sphere with a downward one too."""
    gen = torch.Generator(device=device)
    gen.manual_seed(int(seed))
    dx = 1.0 / max(case["nx"], case["ny"], case["nz"])
    cells = torch.nonzero(_fluid_mask(case, device).reshape(-1)).reshape(-1)
    nx, ny = case["nx"], case["ny"]
    idx = (cells % nx, (cells // nx) % ny, cells // (nx * ny))
    if case["kind"] == "sdf":  # the order that a stepped scene has: by 8^3 blocks of cells
        block = (idx[0] >> 3) + ((idx[1] >> 3) << 8) + ((idx[2] >> 3) << 16)
        order = torch.argsort(block, stable=True)
        idx = tuple(i[order] for i in idx)
    sub = torch.arange(8, device=device)
    pos = []
    for a in range(3):
        s = (sub >> a) & 1
        jit = torch.rand((cells.numel(), 8), generator=gen, device=device, dtype=torch.float32)
        base = (2 * idx[a][:, None] + s[None, :]).to(torch.float64)
        pos.append(((base + jit.double() * 0.999) * (0.5 * dx)).to(torch.float32).reshape(-1))
        del jit, base
    ph = (torch.rand(6, generator=gen, device=device) * (2 * math.pi)).tolist()
    vel = []
    for a in range(3):
        p, q = pos[(a + 1) % 3], pos[(a + 2) % 3]
        vel.append(0.4 * torch.sin(2 * math.pi * p + ph[2 * a])
                   * torch.cos(2 * math.pi * q + ph[2 * a + 1]))
    if case["scene"] in ("drop", "pool"):
        vel[1] = vel[1] - 1.5 * (pos[1] > 0.45 * case["ny"] * dx).to(torch.float32)
    return [t.contiguous() for t in pos + vel]


def _params(case):
    big = max(case["nx"], case["ny"], case["nz"])
    prm = F.default_params(case["nx"], case["ny"], case["nz"])
    prm.dx = 1.0 / big
    prm.skin = 1e-3 / big
    if case.get("precision") == "mixed":  # the benchmark's tolerances
        prm.precision = F.FLIP_PREC_MIXED_IR
        prm.cg_tol = 1e-3
        prm.ir_tol = 1e-8
    prm.warm_start = int(bool(case.get("warm")))
    if case.get("grid_advect"):
        prm.advect_source = F.FLIP_ADVECT_GRID
    if case["kind"] == "oneshot":
        prm.cfl = 3.0
        prm.ppc_min, prm.ppc_max = 3, 12
    return prm


def _batch_scenes(case):
    rnd = np.random.RandomState(case["shape_seed"])
    out = []
    for _ in range(case["count"]):
        n = int(rnd.randint(case["lo"], case["hi"] + 1))
        frac = math.sqrt(rnd.uniform(0.2, 0.5))
        out.append(dict(kind="frame", scene="wide", nx=n, ny=n, nz=n, frac=frac,
                        precision=case["precision"], warm=False, grid_advect=False))
    return out


# ------------------------------------------------------------------ prepare and run

class _Scene:
    """A scene that a program keeps: its particles in creation order, the handle, the stream."""

    def __init__(self, case, seed):
        self.src = _particles(case, seed)
        self.ids = torch.arange(self.src[0].numel(), dtype=torch.int32, device="cuda")
        self.stream = torch.cuda.Stream()
        self.stream.wait_stream(torch.cuda.current_stream())
        self.sim = F.Simulation(_params(case), *self.src, stream=self.stream.cuda_stream)
        self.sizes = _field_sizes(case)

    def load(self):
        """The program's particles go to the library."""
        F.flip_write(self.sim.h, F.PID, self.ids)
        F.flip_write_particles(self.sim.h, *self.src)

    def results(self):
        """Positions and velocities in creation order, projected face velocities, pressure."""
        n = self.src[0].numel()
        with torch.cuda.stream(self.stream):
            raw = [torch.empty(n, dtype=torch.float32, device="cuda") for _ in range(6)]
            ids = torch.empty(n, dtype=torch.int32, device="cuda")
            F.flip_read_particles(self.sim.h, *raw, ids=ids)
            where = ids.long()
            parts = [torch.empty_like(a).index_copy_(0, where, a) for a in raw]
            return parts + _read_fields(self.sim, self.sizes)


def _field_sizes(case):
    n = (case["nx"], case["ny"], case["nz"])
    faces = [(n[0] + (d == 0)) * (n[1] + (d == 1)) * (n[2] + (d == 2)) for d in range(3)]
    return faces + [n[0] * n[1] * n[2]]


def _read_fields(sim, sizes):
    return [sim.read(f, torch.empty(s, dtype=torch.float32, device="cuda"))
            for f, s in zip(FIELDS, sizes)]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "frame":
        return dict(kind=kind, scene=_Scene(case, seed))
    if kind == "oneshot":
        return dict(kind=kind, src=_particles(case, seed), params=_params(case),
                    stream=torch.cuda.Stream(), sizes=_field_sizes(case))
    if kind == "batch":
        scenes = [_Scene(c, seed + 7919 * k) for k, c in enumerate(_batch_scenes(case))]
        return dict(kind=kind, scenes=scenes, batch=F.Batch(len(scenes)))
    if kind == "solve":
        typ, b = _solve_inputs(case, seed)
        return dict(kind=kind, type=typ, b=b, p=torch.empty_like(b),
                    params=F.default_params(case["nx"], case["ny"], case["nz"]))
    if kind == "sdf":
        scene = _Scene(case, seed)
        surf = F.Surface(F.surface_default_params(scene.sim.params), scene.stream.cuda_stream)
        corners = (case["nx"] + 1) * (case["ny"] + 1) * (case["nz"] + 1)
        return dict(kind=kind, scene=scene, surf=surf, corners=corners)
    return dict(kind=kind, phi=_mesh_field(case, seed), surf=F.Surface(_surface_params(case)))


def run(state):
    kind = state["kind"]
    if kind == "frame":
        s = state["scene"]
        s.load()
        s.sim.step(STEPS)
        return s.results()
    if kind == "oneshot":
        st = state["stream"]
        with F.Simulation(state["params"], *state["src"], stream=st.cuda_stream) as sim:
            sim.step(STEPS)
            with torch.cuda.stream(st):
                return _read_fields(sim, state["sizes"])
    if kind == "batch":
        scenes = state["scenes"]
        for s in scenes:
            s.load()
        state["batch"].step([s.sim for s in scenes], STEPS)
        per_scene = [s.results() for s in scenes]
        return [torch.cat(parts) for parts in zip(*per_scene)]
    if kind == "solve":
        F.flip_solve_pressure(state["params"], state["type"], state["b"], state["p"])
        return state["p"]
    if kind == "sdf":
        s, surf = state["scene"], state["surf"]
        surf.sdf(s.sim)
        with torch.cuda.stream(s.stream):
            phi = torch.empty(state["corners"], dtype=torch.float32, device="cuda")
        return _surface_read(surf, F.SURF_FIELD, phi)
    surf, phi = state["surf"], state["phi"]
    _ok(F.lib().flip_surface_set_field(surf.h, phi.data_ptr(), 1))
    nv, nt = surf.mesh()
    return [_surface_read(surf, which, torch.empty(shape, dtype=dt, device="cuda"))
            for which, shape, dt in ((F.SURF_VERTICES, (nv, 3), torch.float32),
                                     (F.SURF_NORMALS, (nv, 3), torch.float32),
                                     (F.SURF_TRIANGLES, (nt, 3), torch.int32),
                                     (F.SURF_VERTEX_EDGE, (nv,), torch.int64))]


def _ok(rc):
    if rc:
        raise RuntimeError(F.last_error())


def _surface_read(surf, which, out):
    _ok(F.lib().flip_surface_read(surf.h, which, out.data_ptr(),
                                  out.numel() * out.element_size(), 1))
    return out


# ------------------------------------------------------------------ the other inputs

def _solve_inputs(case, seed):
    """uint8 cell types (fluid below a wavy surface) and a float32 right-hand side."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    ph = (torch.rand(4, generator=gen, device="cuda") * (2 * math.pi)).tolist()
    x = (torch.arange(nx, device="cuda") + 0.5)[None, None, :] / nx
    y = (torch.arange(ny, device="cuda") + 0.5)[None, :, None] / ny
    z = (torch.arange(nz, device="cuda") + 0.5)[:, None, None] / nz
    top = 0.45 + 0.15 * torch.sin(2 * math.pi * x + ph[0]) * torch.cos(2 * math.pi * z + ph[1])
    typ = (y < top).to(torch.uint8).contiguous()
    b = torch.sin(2 * math.pi * (x + y) + ph[2]) * torch.cos(math.pi * (y + z) + ph[3])
    b = b + 0.2 * torch.randn((nz, ny, nx), generator=gen, device="cuda")
    return typ.reshape(-1), b.to(torch.float32).contiguous().reshape(-1)


def _surface_params(case):
    sp = F.FlipSurfaceParams()
    h = 1.0 / max(case["nx"], case["ny"], case["nz"])
    sp.n[0], sp.n[1], sp.n[2] = case["nx"], case["ny"], case["nz"]
    sp.h, sp.radius, sp.search_radius, sp.iso = h, 0.5 * h, 2.0 * h, 0.0
    return sp


def _mesh_field(case, seed):
    """Corner distances to a wavy sphere, roughened by a factor of 0.6 .. 1.4 per corner, x fastest
    (inputs of all seeds cross zero on the same edges)."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    n = (case["nx"], case["ny"], case["nz"])
    h = 1.0 / max(n)
    ax = [torch.arange(a + 1, device="cuda", dtype=torch.float32) * h for a in n]
    x, y, z = ax[0][None, None, :], ax[1][None, :, None], ax[2][:, None, None]
    c = [0.5 * a * h for a in n]
    r = torch.sqrt((x - c[0]) ** 2 + (y - c[1]) ** 2 + (z - c[2]) ** 2)
    wave = torch.sin(23 * x + 1) * torch.sin(31 * y + 2) * torch.sin(27 * z + 3)
    phi = r - case["radius"] * min(n) * h - 0.04 * wave
    phi = phi * (0.6 + 0.8 * torch.rand(r.shape, generator=gen, device="cuda"))
    return phi.to(torch.float32).contiguous().reshape(-1)


# ------------------------------------------------------------------ what a pass needs

def _n_particles(case):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    return 8 * int(_fluid_mask(case, dev).sum())


def work(case):
    """Bytes and operations of one pass.  A step reads and writes a particle's position and
    velocity once (48 B) and takes about 220 operations per particle (three trilinear splats of a
    value and a weight, three trilinear reads of two values, the blend); the fields that come back
    are written once.  The solve's iterations, whose number the input decides, are not counted."""
    kind = case["kind"]
    if kind in ("frame", "oneshot"):
        n = _n_particles(case)
        return dict(bytes=48.0 * n * STEPS + 4.0 * sum(_field_sizes(case)),
                    flops=220.0 * n * STEPS)
    if kind == "batch":
        each = [work(c) for c in _batch_scenes(case)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    if kind == "solve":
        cells = case["nx"] * case["ny"] * case["nz"]
        return dict(bytes=9.0 * cells, flops=20.0 * cells)
    if kind == "sdf":
        corners = (case["nx"] + 1) * (case["ny"] + 1) * (case["nz"] + 1)
        n = _n_particles(case)
        # a particle lies in the balls of 4/3 pi 2^3 = 33.5 corners, about 17 operations each
        return dict(bytes=12.0 * n + 4.0 * corners, flops=33.5 * 17.0 * n)
    corners = (case["nx"] + 1) * (case["ny"] + 1) * (case["nz"] + 1)
    area = 4 * math.pi * (case["radius"] * min(case["nx"], case["ny"], case["nz"])) ** 2
    nv = 1.6 * area  # crossing edges of a wavy sphere of that area in cell faces
    return dict(bytes=4.0 * corners + nv * (32.0 + 24.0), flops=60.0 * nv)


# ------------------------------------------------------------------ the same in 64 bits

EXACT_PARTICLES = 45_000_000  # more take too long here


def exact(case, seed):
    kind = case["kind"]
    if kind == "oneshot":  # the reseeded particles come from the library's own generator
        return None
    if kind == "frame":
        return None if _n_particles(case) > EXACT_PARTICLES else _exact_frame(case, seed)
    if kind == "batch":
        cases = _batch_scenes(case)
        if sum(_n_particles(c) for c in cases) > EXACT_PARTICLES:
            return None
        per_scene = [_exact_frame(c, seed + 7919 * k) for k, c in enumerate(cases)]
        return [torch.cat(parts) for parts in zip(*per_scene)]
    if kind == "solve":
        typ, b = _solve_inputs(case, seed)
        n = (case["nx"], case["ny"], case["nz"])
        h = 1.0 / max(n)
        shape = (n[2], n[1], n[0])
        return _exact_pressure((typ == 1).reshape(shape), b.double().reshape(shape),
                               DT / (h * h)).reshape(-1)
    if kind == "sdf":
        return None if _n_particles(case) > EXACT_PARTICLES else _exact_sdf(case, seed)
    return _exact_mesh(case, seed)


def _exact_pressure(fluid, b, scale):
    """A p = b by conjugate gradients in 64 bits: scale times the 7-point operator, p = 0 in air,
    walls dropped."""
    f = fluid.double()
    count = torch.full_like(f, 6.0)
    for a in range(3):
        count.narrow(a, 0, 1).sub_(1.0)
        count.narrow(a, f.shape[a] - 1, 1).sub_(1.0)

    def apply(v):
        s = count * v
        for a in range(3):
            m = f.shape[a] - 1
            s.narrow(a, 0, m).sub_(v.narrow(a, 1, m))
            s.narrow(a, 1, m).sub_(v.narrow(a, 0, m))
        return s * f * scale

    inv = f / (count * scale)
    x = torch.zeros_like(f)
    r = b * f
    z = r * inv
    p = z.clone()
    rz = (r * z).sum()
    stop = 1e-13 * float(r.norm())
    for it in range(20000):
        q = apply(p)
        alpha = rz / (p * q).sum().clamp_min(1e-300)
        x.add_(alpha * p)
        r.sub_(alpha * q)
        if it % 16 == 15 and float(r.norm()) <= stop:
            break
        z = r * inv
        new = (r * z).sum()
        p = z + (new / rz.clamp_min(1e-300)) * p
        rz = new
    return x


def _exact_frame(case, seed):
    """The steps in 64 bits on the float32 state that a step starts from and ends with."""
    n = (case["nx"], case["ny"], case["nz"])
    big = max(n)
    h = 1.0 / big
    skin = 1e-3 / big
    part = [t.double() for t in _particles(case, seed)]
    scale = DT / (h * h)
    for _ in range(STEPS):
        pos, vel = part[:3], part[3:]
        cell = [torch.floor(pos[a] * big).clamp_(0, n[a] - 1).long() for a in range(3)]
        flat = cell[0] + n[0] * (cell[1] + n[1] * cell[2])
        fluid = torch.zeros(n[0] * n[1] * n[2], dtype=torch.bool, device=flat.device)
        fluid[flat] = True
        fluid = fluid.reshape(n[2], n[1], n[0])

        def nodes(d):
            """(face index, weight) of the eight nodes of component d around every particle."""
            dim = [n[a] + (a == d) for a in range(3)]
            base, frac = [], []
            for a in range(3):
                if a == d:
                    c = cell[a]
                    f = (pos[a] * big - c).clamp(0.0, 1.0)
                else:
                    g = (pos[a] * big - 0.5).clamp(0.0, n[a] - 1.0)
                    c = torch.floor(g).clamp_max(n[a] - 2.0).long()
                    f = g - c
                base.append(c)
                frac.append(f)
            for q in range(8):
                o = [(q >> a) & 1 for a in range(3)]
                w = 1.0
                for a in range(3):
                    w = w * (frac[a] if o[a] else 1.0 - frac[a])
                yield ((base[0] + o[0]) + dim[0] * ((base[1] + o[1]) + dim[1] * (base[2] + o[2])),
                       w)

        old, star = [], []
        for d in range(3):
            shape = [n[2] + (d == 2), n[1] + (d == 1), n[0] + (d == 0)]
            num = torch.zeros(shape[0] * shape[1] * shape[2], dtype=torch.float64,
                              device=flat.device)
            den = torch.zeros_like(num)
            for i, w in nodes(d):
                num.index_add_(0, i, w * vel[d])
                den.index_add_(0, i, w)
            u = torch.where(den > 0, num / den.clamp_min(1e-300), 0.0).reshape(shape)
            old.append(u)
            s = u + (GRAVITY * DT if d == 1 else 0.0)
            s.narrow(2 - d, 0, 1).zero_()
            s.narrow(2 - d, n[d], 1).zero_()
            star.append(s)
        div = sum(star[d].narrow(2 - d, 1, n[d]) - star[d].narrow(2 - d, 0, n[d])
                  for d in range(3)) * big
        p = _exact_pressure(fluid, -div * fluid, scale)
        new = []
        for d in range(3):
            u = star[d].clone()
            m = n[d] - 1
            u.narrow(2 - d, 1, m).sub_((p.narrow(2 - d, 1, m) - p.narrow(2 - d, 0, m)) * (DT * big))
            new.append(u)
        out_pos, out_vel = [], []
        for d in range(3):
            un, de = new[d].reshape(-1), (new[d] - old[d]).reshape(-1)
            pic = torch.zeros_like(pos[0])
            change = torch.zeros_like(pos[0])
            for i, w in nodes(d):
                pic.add_(w * un[i])
                change.add_(w * de[i])
            v = FLIP_RATIO * (vel[d] + change) + (1.0 - FLIP_RATIO) * pic
            x = pos[d] + DT * (pic if case.get("grid_advect") else v)
            out_pos.append(x.clamp(skin, n[d] * h - skin))
            out_vel.append(v)
        part = [t.float().double() for t in out_pos + out_vel]
    return out_pos + out_vel + [u.reshape(-1) for u in new] + [p.reshape(-1)]


def _exact_sdf(case, seed):
    """The blobby distance of every corner: each particle is added to the 4^3 corners around it,
    the only ones that can be closer than R = 2 h."""
    n = (case["nx"], case["ny"], case["nz"])
    h = 1.0 / max(n)
    radius, reach = 0.5 * h, 2.0 * h
    pos = [t.double() for t in _particles(case, seed)[:3]]
    c = [a + 1 for a in n]
    sums = [torch.zeros(c[0] * c[1] * c[2], dtype=torch.float64, device="cuda") for _ in range(4)]
    base = [torch.floor(p / h).long() for p in pos]
    for q in range(64):
        at = [base[a] + ((q >> (2 * a)) & 3) - 1 for a in range(3)]
        e = [pos[a] - at[a] * h for a in range(3)]
        s2 = (e[0] ** 2 + e[1] ** 2 + e[2] ** 2) / (reach * reach)
        k = (1.0 - s2).clamp_min(0.0) ** 3
        keep = (k > 0)
        for a in range(3):
            keep &= (at[a] >= 0) & (at[a] < c[a])
        i = (at[0] + c[0] * (at[1] + c[1] * at[2]))[keep]
        k = k[keep]
        sums[0].index_add_(0, i, k)
        for a in range(3):
            sums[1 + a].index_add_(0, i, k * e[a][keep])
    w = sums[0]
    mean = torch.sqrt(sums[1] ** 2 + sums[2] ** 2 + sums[3] ** 2) / w.clamp_min(1e-300)
    return torch.where(w > 0, mean - radius, reach - radius)


def _exact_mesh(case, seed):
    """The vertices, by grid edge (3 * corner + axis); the normals follow from triangles, which
    are whole numbers with no such value."""
    n = (case["nx"], case["ny"], case["nz"])
    h = 1.0 / max(n)
    c = [a + 1 for a in n]
    phi = _mesh_field(case, seed).double().reshape(c[2], c[1], c[0])
    ids, verts = [], []
    for a in range(3):
        lo, hi = phi.narrow(2 - a, 0, n[a]), phi.narrow(2 - a, 1, n[a])
        k, j, i = torch.nonzero((lo < 0) != (hi < 0), as_tuple=True)
        t = -lo[k, j, i] / (hi[k, j, i] - lo[k, j, i])
        v = torch.stack([i, j, k], 1).double()
        v[:, a] += t
        ids.append(3 * (i + c[0] * (j + c[1] * k)) + a)
        verts.append(v * h)
    order = torch.argsort(torch.cat(ids))
    return [torch.cat(verts)[order], None, None, None]
