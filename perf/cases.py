"""Workloads of the library as its users run them, for timing: listed() gives fixed ones,
draw() others of the same ranges, prepare() what a program has in hand before the call,
run() one pass through the public entry points, work() the bytes and operations of a pass
and exact() the same results in 64 bits by plain torch.

Every context of a process queues on one stream (`stream()`), as a program with one
simulation loop does. The library returns FP64 arrays whatever it computes in; run() hands
the values on in the type they were computed in (FP32) or are stored in (the density and
velocity of a 16-bit lattice), positions in FP64 as the library integrates them.
"""
import math

import numpy as np
import torch

import paper_1901_09745_gb300 as P

# Contact law of the coupled workloads (lattice units), as in the benchmark and the tests.
DEM = dict(E=2.0, poisson=0.3, gamma=2e-4, density=3.0, mu_f=0.3, theta_crit=0.01, alpha_n=0.3, k_t_scale=1.0,
           eta_t_scale=1.0)
PERIODIC, WALL, OPEN, INFLOW = 0, 1, 2, 3
TYPES = {"f64": torch.float64, "f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
BYTES = {"f64": 8, "f32": 4, "f16": 2, "bf16": 2}


def case(name, kind, lattice, n, bc, storage, particles, radii, steps, tau=0.7, force=1e-6, band=1.0, psc=0, **more):
    """One workload. kind: "static" (fixed particles), "coupled" (fluid step and DEM call),
    "driven" (the caller moves the particles), "inlet" (flow past a fixed sphere), "dem"
    (contacts only), "buffers" (one step on the caller's own arrays), "adjoint". band: the
    part of the slowest axis that holds the particles."""
    c = dict(kind=kind, lattice=lattice, nx=n[0], ny=n[1], nz=n[2], bx=bc[0], by=bc[1], bz=bc[2], storage=storage,
             particles=particles, rmin=float(radii[0]), rmax=float(radii[1]), steps=steps, tau=tau, force=force,
             band=band, psc=psc, substeps=10, packing="random", gravity=0.0, gamma=2e-4, every=0)
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest calls: four fixed discs in a 64 x 64 box, FP64, fields and forces read every step
        case("discs_64", "static", 9, (64, 64, 1), (0, 0, 0), "f64", 4, (6.5, 6.5), 1, tau=0.8),
        # a fixed array of discs in a ragged walled channel, read every ten steps
        case("channel_ragged", "static", 9, (777, 453, 1), (0, 1, 0), "f32", 500, (4, 8), 10),
        # the headline workload: 2048 x 2048 channel with 5000 mobile discs, coupled to the DEM
        case("channel_2048", "coupled", 9, (2048, 2048, 1), (0, 1, 0), "f32", 5000, (4, 8), 20, force=0.0, band=0.357),
        # the caller moves the discs itself: every step host arrays in, forces back to the host
        case("channel_driven", "driven", 9, (1024, 1024, 1), (0, 1, 0), "f32", 1250, (4, 8), 4, band=0.357),
        # one step on the caller's own device buffers, ragged lattice, moving discs
        case("channel_buffers", "buffers", 9, (1537, 1025, 1), (0, 1, 0), "f32", 1800, (4, 8), 1, band=0.5),
        # a fixed bed of spheres in 3D at solid fraction 0.11
        case("bed_256", "static", 19, (256, 256, 256), (0, 0, 0), "f32", 2000, (6, 6), 10, tau=0.6),
        # the same box at solid fraction 0.3, FP16 storage
        case("bed_256_dense", "static", 19, (256, 256, 256), (0, 0, 0), "f16", 5563, (6, 6), 10, tau=0.6),
        # the largest: 512^3 channel with 50000 mobile spheres, FP16 storage, coupled to the DEM
        case("channel_512", "coupled", 19, (512, 512, 512), (0, 0, 1), "f16", 50000, (3, 8), 5, tau=0.55, gamma=2e-2),
        # drag of one fixed sphere between a velocity inlet and a pressure outlet, open sides
        case("drag", "inlet", 19, (120, 60, 60), (3, 2, 2), "f32", 1, (3, 3), 20, tau=0.572, force=0.0),
        # 500 spheres settling onto a wall
        case("settling", "coupled", 19, (50, 50, 100), (0, 0, 1), "f32", 500, (3, 3), 10, tau=2.0, force=0.0,
             packing="bed", gravity=-5e-4, gamma=2e-3, E=20.0),
        # contacts alone: a bed of 24576 touching spheres under gravity
        case("bed_contacts", "dem", 19, (192, 192, 160), (0, 0, 1), "f16", 24576, (3, 3), 1, force=0.0, packing="bed",
             gravity=-5e-4, gamma=2e-3, E=20.0),
        # gradient of the drag of 200 fixed spheres in a 128^3 box
        case("gradient_128", "adjoint", 19, (128, 128, 128), (0, 0, 0), "f32", 200, (5, 5), 20, every=5),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(("static", "static", "static", "coupled", "coupled", "coupled", "driven", "buffers", "inlet", "dem",
                       "adjoint"))
    storage = rng.choice(("f32", "f32", "f32", "f16", "f16", "bf16", "f64"))
    flat = rng.random() < 0.5 and kind not in ("inlet", "dem")
    if kind == "inlet":
        d = rng.choice((5, 6, 7, 8, 9))
        return case(None, kind, 19, (20 * d + rng.randrange(8), 10 * d + rng.randrange(6), 10 * d + rng.randrange(6)),
                    (3, 2, 2), storage, 1, (d / 2, d / 2), rng.randrange(8, 24), tau=rng.uniform(0.56, 0.9), force=0.0)
    if kind == "dem":
        a, b, c = rng.randrange(6, 40), rng.randrange(6, 40), rng.randrange(4, 30)
        return case(None, kind, 19, (6 * a, 6 * b, 6 * c + 20), (0, 0, 1), storage, a * b * c, (3, 3), 1, force=0.0,
                    packing="bed", gravity=-5e-4, gamma=2e-3, E=20.0)
    hi = {"buffers": 2048 if flat else 150, "adjoint": 512 if flat else 128, "driven": 1500 if flat else 160}.get(
        kind, 2048 if flat else 288)
    if storage == "f64":
        hi = int(hi * (0.7 if flat else 0.6))
    n = tuple(size(64 if flat else 40, hi) for _ in range(2 if flat else 3)) + ((1,) if flat else ())
    walls = (0, rng.randrange(2), 0) if flat else (0, 0, rng.randrange(2))
    phi = rng.uniform(0.02, 0.36 if flat else 0.28)
    lo, up = (4, 8) if rng.random() < 0.5 else ((5, 5) if rng.random() < 0.5 else (3, 6))
    mean = (lo * lo + lo * up + up * up) / 3 if flat else (lo + up) * (lo * lo + up * up) / 4
    room = n[0] * n[1] if flat else n[0] * n[1] * n[2]
    particles = max(1, int(phi * room / (mean * (math.pi if flat else 4 * math.pi / 3))))
    if kind == "static" and rng.random() < 0.15:
        particles = 0
    band = 1.0 if rng.random() < 0.5 or walls == (0, 0, 0) or particles == 0 else rng.uniform(0.85, 1.0)
    cells = room * BYTES[storage]
    steps = {"static": max(1, min(10, int(2e8 / cells))), "coupled": max(1, min(10, int(2e8 / cells))),
             "driven": 4, "buffers": 1, "adjoint": max(4, min(20, int(2e8 / cells)))}[kind]
    if kind == "adjoint":
        storage = "f64" if storage == "f64" else "f32"
    return case(None, kind, 9 if flat else 19, n, walls, storage, particles, (lo, up), steps,
                tau=round(rng.uniform(0.55, 1.0), 3), force=rng.choice((0.0, 1e-6)), band=band,
                psc=int(kind == "static" and rng.random() < 0.2), every=rng.randrange(2, 6))


# ------------------------------------------------------------------------------- inputs
_STREAM = []


def stream():
    if not _STREAM:
        _STREAM.append(torch.cuda.Stream())
    return _STREAM[0]


def extent(c):
    return (c["nx"], c["ny"], c["nz"])


def walls(c):
    return (c["bx"], c["by"], c["bz"])


def pack(rng, box, walled, radii, lo, hi):
    """Centres of non-overlapping particles by random sequential addition, largest first."""
    dim = len(box)
    box = np.asarray(box, dtype=np.float64)
    X = np.zeros((len(radii), dim))
    order = np.argsort(-radii, kind="stable")
    for k, i in enumerate(order):
        m = 8
        while True:
            x = lo + rng.random((m, dim)) * (hi - lo)
            ok = np.ones(m, dtype=bool)
            for a in range(dim):
                if walled[a]:
                    ok &= (x[:, a] - radii[i] >= 0.0) & (x[:, a] + radii[i] <= box[a] - 1.0)
            d = x[:, None, :] - X[None, order[:k], :]
            for a in range(dim):
                if not walled[a]:
                    d[..., a] -= box[a] * np.rint(d[..., a] / box[a])
            ok &= ((d * d).sum(-1) >= (radii[i] + radii[order[:k]]) ** 2).all(-1)
            hit = np.flatnonzero(ok)
            if hit.size:
                X[i] = x[hit[0]]
                break
            m *= 2
            if m > 1 << 17:
                raise RuntimeError("the packing is too dense")
    return X


def particles(c, seed):
    """X, U, Om (n x 3) and radii: a random packing of one block of the box, repeated along
    the periodic axes, or a bed of touching spheres on the lower wall."""
    rng = np.random.default_rng(seed)
    n, dim, box = c["particles"], 2 if c["lattice"] == 9 else 3, extent(c)
    if n == 0:
        z = np.zeros((0, 3))
        return z, z, z, np.zeros(0)
    if c["kind"] == "inlet":
        X = np.array([[0.5 * (v - 1) for v in box]]) + rng.uniform(-0.5, 0.5, (1, 3))
        return X, np.zeros((1, 3)), np.zeros((1, 3)), np.full(1, c["rmin"])
    if c["packing"] == "bed":
        r = np.full(n, c["rmin"]) + 0.004
        a, b = int(box[0] // (2 * c["rmin"])), int(box[1] // (2 * c["rmin"]))
        k = np.arange(n)
        X = np.stack([(k % a + 0.5) * box[0] / a, (k // a % b + 0.5) * box[1] / b,
                      c["rmin"] - 0.5 + 2 * c["rmin"] * (k // (a * b))], axis=1)
        X += rng.uniform(-0.01, 0.01, (n, 3))
        U = rng.normal(0.0, 1e-4, (n, 3))
        return X, U, rng.normal(0.0, 1e-5, (n, 3)), r
    walled = [walls(c)[a] != PERIODIC for a in range(dim)]
    copies = [1] * dim
    while n // math.prod(copies) > 800:
        a = max((a for a in range(dim) if not walled[a]), key=lambda a: box[a] / copies[a])
        copies[a] *= 2
    m = -(-n // math.prod(copies))
    block = [box[a] / copies[a] for a in range(dim)]
    r = rng.uniform(c["rmin"], c["rmax"], m)
    lo, hi = np.zeros(dim), np.array(block)
    lo[-1], hi[-1] = (0.5 - 0.5 * c["band"]) * block[-1], (0.5 + 0.5 * c["band"]) * block[-1]
    Xb = pack(rng, block, walled, r, lo, hi)
    shifts = np.stack(np.meshgrid(*[np.arange(k) for k in copies], indexing="ij"), -1).reshape(-1, dim) * np.array(block)
    X = np.zeros((m * len(shifts), 3))
    X[:, :dim] = (Xb[None] + shifts[:, None]).reshape(-1, dim)
    X, r = X[:n], np.tile(r, len(shifts))[:n]
    U, Om = np.zeros((n, 3)), np.zeros((n, 3))
    if c["kind"] in ("coupled", "driven", "buffers"):
        U[:, :dim] = rng.normal(0.0, 1e-3, (n, dim))
        if dim == 2:
            Om[:, 2] = rng.normal(0.0, 1e-3, n) / r
        else:
            Om[:] = rng.normal(0.0, 1e-3, (n, 3)) / r[:, None]
    return X, U, Om, r


def table(lattice):
    """Velocities, weights and opposite directions in the order of the library's header."""
    if lattice == 9:
        e = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0)]
        w = [4 / 9, 1 / 9, 1 / 36]
    else:
        e = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)]
        for p in ((1, 1, 0), (1, -1, 0), (1, 0, 1), (1, 0, -1), (0, 1, 1), (0, 1, -1)):
            e += [p, tuple(-v for v in p)]
        w = [1 / 3, 1 / 18, 1 / 36]
    return e, [w[sum(v * v for v in ei)] for ei in e], [e.index(tuple(-v for v in ei)) for ei in e]


def flow(c, seed):
    """Populations of a smooth flow (velocities of a few hundredths, or the inlet's stream)
    with a little noise: deviations from the weights, FP64, [Q][nz][ny][nx]."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    rng = np.random.default_rng(seed + 1)
    n = extent(c)
    x = [torch.arange(n[a], dtype=torch.float64, device="cuda").reshape([-1 if 2 - a == k else 1 for k in range(3)])
         for a in range(3)]
    dim = 2 if c["lattice"] == 9 else 3
    shape = (n[2], n[1], n[0])
    u = []
    for a in range(3):
        if a >= dim or c["kind"] == "inlet":
            u.append(torch.full((1, 1, 1), 0.04 if c["kind"] == "inlet" and a == 0 else 0.0, dtype=torch.float64, device="cuda"))
            continue
        k, ph = rng.integers(1, 4, 3), rng.uniform(0, 2 * math.pi)
        u.append(0.02 * torch.sin(sum(2 * math.pi * int(k[b]) / n[b] * x[b] for b in range(dim)) + ph))
    e, w, _ = table(c["lattice"])
    uu = sum(v * v for v in u)
    f = torch.empty((len(e),) + shape, dtype=torch.float64, device="cuda")
    for i, ei in enumerate(e):
        eu = sum(ei[a] * u[a] for a in range(3) if ei[a])
        f[i] = w[i] * (3 * eu + 4.5 * eu * eu - 1.5 * uu)
        f[i] += w[i] * 1e-3 * (torch.rand(shape, generator=gen, dtype=torch.float32, device="cuda") - 0.5)
    return f


def body_force(c):
    return (c["force"], 0.0, 0.0)


def dem_values(c):
    v = dict(DEM, gamma=c["gamma"], E=c.get("E", DEM["E"]))
    return dict(v, dt_dem=1.0 / c["substeps"], gravity=(0.0, 0.0, c["gravity"]), adhesive=1)


def prepare(c, seed):
    s = dict(c=c, stream=stream())
    X, U, Om, r = particles(c, seed)
    n = len(r)
    shape = extent(c)[::-1]
    dev = dict(dtype=torch.float64, device="cuda")
    with torch.cuda.stream(s["stream"]):
        if c["kind"] == "buffers":
            s["params"] = params = P.LbmParams()
            params.lattice, params.nx, params.ny, params.nz = c["lattice"], c["nx"], c["ny"], c["nz"]
            params.bc[:], params.tau, params.body_force[:] = walls(c), c["tau"], body_force(c)
            params.storage, params.psc, params.stream = P.STORAGE[c["storage"]], c["psc"], s["stream"].cuda_stream
            scale = 4096.0 if c["storage"] == "f16" else 1.0
            s["f"] = (flow(c, seed) * scale).to(TYPES[c["storage"]])
            s["g"] = torch.empty_like(s["f"])
            s["particles"] = [torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (X, U, Om, r)]
            s["F"], s["T"] = torch.zeros((n, 3), **dev), torch.zeros((n, 3), **dev)
            return s
        s["ctx"] = ctx = P.lbm_create(c["lattice"], *extent(c), bc=walls(c), tau=c["tau"], body_force=body_force(c),
                                      storage=c["storage"], psc=c["psc"], stream=s["stream"].cuda_stream,
                                      inflow=(0.04 if c["bx"] == INFLOW else 0.0, 0.0, 0.0))
        if c["kind"] != "dem":
            f = flow(c, seed)
            for i, w in enumerate(table(c["lattice"])[1]):
                f[i] += w
            P.lbm_set_populations(ctx, f)
            del f
        if c["kind"] == "driven":
            s["moves"] = [X + k * U for k in range(c["steps"])]
            s["U"], s["Om"], s["r"] = U, Om, r
            s["F"] = torch.zeros((c["steps"], n, 3), dtype=torch.float64).pin_memory()
            s["T"] = torch.zeros((c["steps"], n, 3), dtype=torch.float64).pin_memory()
        if n:
            P.lbm_set_particles(ctx, X, U, Om, r)
        if c["kind"] in ("coupled", "dem"):
            s["dem"] = P.dem_create(ctx, **dem_values(c))
            s["X"], s["U"], s["Om"] = (torch.zeros((n, 3), **dev) for _ in range(3))
        if c["kind"] != "driven":
            s["F"], s["T"] = torch.zeros((n, 3), **dev), torch.zeros((n, 3), **dev)
        if c["kind"] not in ("dem", "adjoint"):
            s["rho"], s["u"] = torch.zeros(shape, **dev), torch.zeros(shape + (3,), **dev)
    return s


# -------------------------------------------------------------------------------- a pass
def run(s):
    c = s["c"]
    wide = torch.float64 if c["storage"] == "f64" else torch.float32
    with torch.cuda.stream(s["stream"]):
        if c["kind"] == "buffers":
            P.lbm_psc_step_noalloc(s["params"], s["f"], s["g"], *s["particles"], s["F"], s["T"])
            s["f"], s["g"] = s["g"], s["f"]
            return dict(f=s["f"], F=s["F"].to(wide), T=s["T"].to(wide))
        ctx = s["ctx"]
        if c["kind"] == "adjoint":
            J, dX, dF = P.lbm_adjoint_drag(ctx, c["steps"], c["every"])
            t = np.float64 if c["storage"] == "f64" else np.float32
            return dict(J=np.full(1, J, dtype=t), dX=dX.astype(t), dF=dF.astype(t))
        if c["kind"] == "driven":
            for k, X in enumerate(s["moves"]):
                P.lbm_set_particles(ctx, X, s["U"], s["Om"], s["r"])
                P.lbm_step(ctx, 1)
                P.lbm_get_forces(ctx, s["F"][k], s["T"][k])
        elif c["kind"] == "coupled":
            P.lbm_coupled_step(ctx, s["dem"], c["steps"], c["substeps"])
        elif c["kind"] == "dem":
            P.dem_step(s["dem"], c["substeps"] * c["steps"])
        else:
            P.lbm_step(ctx, c["steps"])
        out = {}
        if c["kind"] in ("coupled", "dem"):
            P.dem_get_particles(s["dem"], s["X"], s["U"], s["Om"])
            out.update(X=s["X"], U=s["U"].to(wide), Om=s["Om"].to(wide))
        if c["kind"] not in ("dem", "driven") and c["particles"]:
            P.lbm_get_forces(ctx, s["F"], s["T"])
        if c["kind"] != "dem":
            P.lbm_get_macro(ctx, s["rho"], s["u"])
            t = TYPES[c["storage"]]
            out.update(F=s["F"].to(wide), T=s["T"].to(wide), rho=s["rho"].to(t), u=s["u"].to(t))
        return out


def work(c):
    """Per lattice step the state is read and written once (the gradient: once more forward,
    and the state and two adjoint fields backward); per DEM sub-step the particles' state and
    two spring histories of each of their contacts."""
    q, cells, n = c["lattice"], c["nx"] * c["ny"] * c["nz"], c["particles"]
    field = q * cells * BYTES[c["storage"]]
    flop = (150 if q == 9 else 340) * cells
    steps = c["steps"]
    contacts = n * (6 if c["packing"] == "bed" else 1)
    sub = dict(bytes=n * (2 * 72 + 48) + contacts * 2 * 32, flops=n * 60 + contacts * 250)
    if c["kind"] == "dem":
        return {k: v * steps * c["substeps"] for k, v in sub.items()}
    if c["kind"] == "adjoint":
        return dict(bytes=7 * field * steps, flops=4 * flop * steps)
    b = 2 * field * steps + n * 80 + n * 48
    if c["kind"] != "buffers":
        b += field + 32 * cells          # density and velocity, FP64
    f = flop * steps
    if c["kind"] == "coupled":
        b += sub["bytes"] * c["substeps"] * steps
        f += sub["flops"] * c["substeps"] * steps
    if c["kind"] == "driven":
        b += (steps - 1) * n * (80 + 48)
    return dict(bytes=b, flops=f)


# ---------------------------------------------------------------- the same in 64 bits
class Fluid:
    """One lattice step as the header states it, on whole fields in FP64. `g` holds what the
    cells stored after their collision (deviations from the weights)."""

    def __init__(self, c):
        self.c, self.n, self.bc = c, extent(c), walls(c)
        self.dim = 2 if c["lattice"] == 9 else 3
        self.e, self.w, self.o = table(c["lattice"])

    def face(self, f, a, hi):
        return f.select(2 - a, self.n[a] - 1 if hi else 0)

    def unpull(self, f):
        """What the cells must have stored for the pull to give f."""
        g = torch.empty_like(f)
        for i, e in enumerate(self.e):
            g[i] = torch.roll(f[i], [-e[2], -e[1], -e[0]], (0, 1, 2))
            for kinds, src in (((OPEN, INFLOW), i), ((WALL,), self.o[i])):
                for a in range(self.dim):
                    if e[a] and self.bc[a] in kinds:
                        self.face(g[i], a, e[a] > 0).copy_(self.face(f[src], a, e[a] > 0))
        return g

    def pull(self, g):
        f = []
        for i, e in enumerate(self.e):
            v = g[i]
            for a in range(self.dim):
                if e[a]:
                    r = torch.roll(v, e[a], 2 - a)
                    if self.bc[a] == OPEN:           # the face keeps its own value
                        self.face(r, a, e[a] < 0).copy_(self.face(v, a, e[a] < 0))
                    v = r
            for a in range(self.dim):
                if e[a] and self.bc[a] == WALL:
                    v = v.clone() if v is g[i] else v
                    self.face(v, a, e[a] < 0).copy_(self.face(g[self.o[i]], a, e[a] < 0))
            f.append(v)
        if self.bc[0] == INFLOW:
            for hi in (0, 1):
                s = -1 if hi == 0 else 1             # the known side of the face
                sd = sum((1 if e[0] == 0 else 2) * self.face(f[i], 0, hi) for i, e in enumerate(self.e) if e[0] in (0, s))
                flux = sd if hi else (1 + sd) / (1 - 0.04) * 0.04
                for i, e in enumerate(self.e):
                    if e[0] == -s:
                        self.face(f[i], 0, hi).copy_(self.face(f[self.o[i]], 0, hi) + 6 * self.w[i] * (e[0] if hi else 1) * flux)
        return f

    def moments(self, f, F):
        drho = sum(f)
        j = [sum(e[a] * f[i] for i, e in enumerate(self.e) if e[a]) if a < self.dim else torch.zeros_like(drho)
             for a in range(3)]
        return drho, j, [(j[a] + 0.5 * F[a]) / (1 + drho) for a in range(3)]

    def shells(self, X, r, Xd=None):
        """Every (particle, cell) with a solid fraction: particle, cell, fraction, arm."""
        dim, dev = self.dim, X.device
        fr = height(dim, r)
        k = int(math.ceil(float(r.max()) + 1.0))
        ax = torch.arange(-k, k + 2, device=dev)
        grid = torch.stack(torch.meshgrid(*[ax] * dim, indexing="ij"), -1).reshape(-1, dim)
        n = torch.tensor(self.n[:dim], device=dev)
        per = torch.tensor([self.bc[a] == PERIODIC for a in range(dim)], device=dev)
        got = []
        for b in range(0, len(r), 2000):
            x = X[b:b + 2000, :dim]
            cell = torch.floor(x).long()[:, None] + grid
            d = cell.double() - x[:, None]
            dist = d.square().sum(-1).sqrt()
            inside = ((cell >= 0) & (cell < n) | per).all(-1)
            rr = r[b:b + 2000, None]
            p, q = torch.nonzero(inside & (dist < rr + 1.0), as_tuple=True)
            at = torch.remainder(cell[p, q], n)
            idx = at[:, 0] + self.n[0] * (at[:, 1] + (self.n[1] * at[:, 2] if dim == 3 else 0))
            if Xd is not None:                       # differentiable in the positions
                arm = d[p, q] + (x[p] - Xd[b + p, :dim])
            else:
                arm = d[p, q]
            dist, rp = arm.square().sum(-1).sqrt(), r[b + p]
            eps = torch.where(dist <= rp - 1.0, torch.ones_like(dist), (fr[b + p] - (dist - rp)).clamp(0, 1))
            arm = torch.nn.functional.pad(arm, (0, 3 - dim))
            keep = eps.detach() > 0
            got.append((b + p[keep], idx[keep], eps[keep], arm[keep]))
        return [torch.cat(v) for v in zip(*got)]

    def collide(self, f, F, shell=None, U=None, Om=None):
        """Post-collision field, force and torque per particle."""
        c, tmh = self.c, self.c["tau"] - 0.5
        shape = f[0].shape
        drho, j, u = self.moments(f, F)
        rho = 1 + drho
        Ft = None
        B = torch.zeros_like(drho)
        m, M = [B] * 3, {}
        if shell is not None:
            p, idx, eps, arm = shell
            cells = drho.numel()
            add = lambda v: torch.zeros(cells, dtype=torch.float64, device=v.device).index_add(0, idx, v).reshape(shape)
            us = U[p] + torch.linalg.cross(Om[p], arm) if U is not None else None
            if c["psc"] == 0:
                sum_eps = add(eps)
                en = sum_eps.clamp(max=1.0)
                B = en * tmh / ((1 - en) + tmh)
                cB = B / torch.where(sum_eps > 0, sum_eps, torch.ones_like(sum_eps))
                wt = eps * cB.reshape(-1)[idx]
                wf = wt
            else:
                wt = eps * tmh / ((1 - eps) + tmh)
                B = add(wt)
                wf = B.reshape(-1)[idx]
            if us is not None:
                m = [add(wt * us[:, a]) if a < self.dim else m[a] for a in range(3)]
                M = {(a, b): add(wt * us[:, a] * us[:, b]) for a in range(self.dim) for b in range(a, self.dim)}
            one = [F[a] / 2 - j[a].reshape(-1)[idx] + (rho.reshape(-1)[idx] * us[:, a] if us is not None else 0) for a in range(3)]
            dP = torch.stack([wf * v for v in one], 1)
            if self.dim == 2:
                dP = dP * torch.tensor([1.0, 1.0, 0.0], dtype=torch.float64, device=dP.device)
            n = self.count
            zero = lambda: torch.zeros((n, 3), dtype=torch.float64, device=dP.device)
            Ft = (-zero().index_add(0, p, dP), -zero().index_add(0, p, torch.linalg.cross(arm, dP)))
        uu = sum(v * v for v in u)
        uF = sum(u[a] * F[a] for a in range(3))
        tr = sum(M[a, a] for a in range(self.dim)) if M else 0.0
        om, guo = 1.0 / c["tau"], 1.0 - 0.5 / c["tau"]
        out = []
        for i, e in enumerate(self.e):
            w, o = self.w[i], self.o[i]
            axes = [a for a in range(3) if e[a]]
            eu = sum((e[a] * u[a] for a in axes), torch.zeros((), dtype=torch.float64, device=drho.device))
            eF = sum(e[a] * F[a] for a in axes)
            even = w * (drho + rho * (4.5 * eu * eu - 1.5 * uu))
            odd = w * rho * 3 * eu
            v = f[i] + (1 - B) * (guo * w * (3 * (eF - uF) + 9 * eu * eF) - om * (f[i] - even - odd))
            if shell is not None:
                v = v + B * (f[o] - f[i] - even + odd) + w * B * drho
                if M:
                    em = sum(e[a] * m[a] for a in axes)
                    eMe = sum(e[a] * e[b] * M[min(a, b), max(a, b)] for a in axes for b in axes)
                    v = v + w * rho * (3 * em + 4.5 * eMe - 1.5 * tr)
            out.append(v)
        return torch.stack(out), Ft

    count = 0


def height(dim, r):
    """f(r) of the linear approximation: the solid part of the cell a particle's edge cuts."""
    if dim == 2:
        s = (r * r - 0.25).sqrt()
        va = 0.5 * s + r * r * torch.atan(0.5 / s)
    else:
        r2 = r * r
        s = (r2 - 0.5).sqrt()
        va = ((1 / 12 - r2) * torch.atan(0.5 * s / (0.5 - r2)) + s / 3 + (r2 - 1 / 12) * torch.atan(0.5 / s)
              - 4 / 3 * r2 * r * torch.atan(0.25 / (r * s)))
    return va - r + 0.5


class Contacts:
    """The contact law of the header (JKR, friction, twisting and rolling springs) in FP64."""

    def __init__(self, c, X, r):
        self.c, self.v, self.r = c, dem_values(c), r
        self.dim = 2 if c["lattice"] == 9 else 3
        self.n = torch.tensor(extent(c), dtype=torch.float64, device=r.device)
        self.per = torch.tensor([b == PERIODIC for b in walls(c)], device=r.device)
        rho = self.v["density"]
        self.m = rho * math.pi * r ** 2 if self.dim == 2 else rho * 4 / 3 * math.pi * r ** 3
        self.I = (0.5 if self.dim == 2 else 0.4) * self.m * r * r
        i, j = [], []
        for b in range(0, len(r), 1024):
            d = self.image(X[None] - X[b:b + 1024, None]).square().sum(-1)
            near = d < (r[None] + r[b:b + 1024, None] + 1.0) ** 2
            p, q = torch.nonzero(near, as_tuple=True)
            p = p + b
            i.append(p[p < q])
            j.append(q[p < q])
        self.i, self.j = torch.cat(i), torch.cat(j)
        self.pair = self.springs(len(self.i))
        self.wall = {a: self.springs(len(r)) for a in range(self.dim) if not self.per[a]}

    def springs(self, k):
        z = lambda *s: torch.zeros((k,) + s, dtype=torch.float64, device=self.r.device)
        return dict(s=z(3), t=z(), r=z(3), on=z().bool())

    def image(self, d):
        return torch.where(self.per, d - self.n * torch.round(d / self.n), d)

    def law(self, h, gap, nv, ri, rj, R, ms, vi, vj, oi, oj):
        v = self.v
        Es = v["E"] / (2 * (1 - v["poisson"] ** 2))
        Gs = v["E"] / (4 * (2 - v["poisson"]) * (1 + v["poisson"]))
        FC = 3 * math.pi * v["gamma"] * R
        a0 = (9 * math.pi * v["gamma"] * R * R / Es) ** (1 / 3)
        on = (gap >= 0) | h["on"] & (gap > -a0 * a0 / (2 * 6 ** (1 / 3) * R))
        sc = 6 ** (-1 / 3)
        lhs = (gap * R / a0 ** 2 + 0.5 * sc).clamp(min=0)
        x = torch.minimum((lhs / (6 * sc * sc)).sqrt(), lhs ** 0.25)
        for _ in range(60):
            slope = x * (12 * sc * sc + 12 * sc * x + 4 * x * x)
            x = (x - (x * x * (6 * sc * sc + 4 * sc * x + x * x) - lhs) / slope.clamp(min=1e-300)).clamp(min=0)
        s = sc + x
        a = s * s * a0
        Fe, kr = 4 * FC * (s ** 6 - s ** 3), 4 * FC * s ** 3
        eN = v["alpha_n"] * (ms * 2 * Es * a).sqrt()
        kT, eT, dt = v["k_t_scale"] * 8 * Gs * a, v["eta_t_scale"] * eN, v["dt_dem"]
        cross = torch.linalg.cross
        rel = (vi + cross(oi, ri[:, None] * nv)) - (vj + cross(oj, -rj[:, None] * nv))
        vn = (rel * nv).sum(-1)
        vt = rel - vn[:, None] * nv

        def turned(q):
            p = q - (q * nv).sum(-1, keepdim=True) * nv
            a, b = q.norm(dim=-1, keepdim=True), p.norm(dim=-1, keepdim=True)
            return torch.where(b > 0, p * a / b.clamp(min=1e-300), p)

        cap = v["mu_f"] * (Fe + 2 * FC).abs()
        xs = turned(h["s"]) + vt * dt
        Ft = -kT[:, None] * xs - eT[:, None] * vt
        mag = Ft.norm(dim=-1)
        slip = mag > cap
        Ft = torch.where(slip[:, None], Ft * (cap / mag.clamp(min=1e-300))[:, None], Ft)
        xs = torch.where(slip[:, None], -Ft / kT[:, None], xs)
        omr = oi - oj
        spin = (omr * nv).sum(-1)
        xt = h["t"] + spin * dt
        kt = kT * a * a * 0.5
        Mt = -kt * xt - eT * a * a * 0.5 * spin
        capt = 3 * math.pi / 16 * a * cap
        slip = Mt.abs() > capt
        Mt = torch.where(slip, torch.sign(Mt) * capt, Mt)
        xt = torch.where(slip, -Mt / kt, xt)
        xr = turned(h["r"]) + (R * dt)[:, None] * cross(nv, omr)
        Mr = kr[:, None] * cross(nv, xr)
        mag, capr = Mr.norm(dim=-1), kr * v["theta_crit"] * R
        slip = mag > capr
        back = torch.where(slip, capr / mag.clamp(min=1e-300), torch.ones_like(mag))[:, None]
        Mr, xr = Mr * back, xr * back
        k = on[:, None].double()
        h.update(s=xs * k, t=xt * on, r=xr * k, on=on)
        force = (-(Fe + eN * vn)[:, None] * nv + Ft) * k
        arm = cross(nv, Ft) * k                      # times each side's radius
        torque = (Mt[:, None] * nv + Mr) * k
        if self.dim == 2:
            force, arm, torque = force * self.flat, arm * (1 - self.flat), torque * (1 - self.flat)
        return force, arm, torque

    def step(self, X, U, Om, F, T):
        r, m, dt = self.r, self.m, self.v["dt_dem"]
        self.flat = torch.tensor([1.0, 1.0, 0.0], dtype=torch.float64, device=X.device)
        g = torch.tensor(self.v["gravity"], dtype=torch.float64, device=X.device)
        f, t = F.clone(), T.clone()
        i, j = self.i, self.j
        if len(i):
            d = self.image(X[j] - X[i])
            dist = d.norm(dim=-1)
            force, arm, torque = self.law(self.pair, r[i] + r[j] - dist, d / dist[:, None], r[i], r[j],
                                          r[i] * r[j] / (r[i] + r[j]), m[i] * m[j] / (m[i] + m[j]), U[i], U[j], Om[i], Om[j])
            f = f.index_add(0, i, force).index_add(0, j, -force)
            t = t.index_add(0, i, arm * r[i, None] + torque).index_add(0, j, arm * r[j, None] - torque)
        for a, h in self.wall.items():
            low = X[:, a] < 0.5 * (self.n[a] - 1)
            nv = torch.zeros_like(X)
            nv[:, a] = torch.where(low, -1.0, 1.0).double()
            dist = torch.where(low, X[:, a] + 0.5, self.n[a] - 0.5 - X[:, a])
            zero = torch.zeros_like(U)
            force, arm, torque = self.law(h, r - dist, nv, r, torch.zeros_like(r), r, m, U, zero, Om, zero)
            f, t = f + force, t + arm * r[:, None] + torque
        if self.dim == 2:
            U = U + dt * (f / m[:, None] + g) * self.flat
            Om = Om + dt * t / self.I[:, None] * (1 - self.flat)
        else:
            U, Om = U + dt * (f / m[:, None] + g), Om + dt * t / self.I[:, None]
        X = X + dt * U
        return torch.where(self.per, X - self.n * torch.floor(X / self.n), X) if self.dim == 3 else torch.cat(
            [torch.where(self.per, X - self.n * torch.floor(X / self.n), X)[:, :2], X[:, 2:]], 1), U, Om


def exact(c, seed):
    # the largest would take too long
    if c["nx"] * c["ny"] * c["nz"] > 3e7:
        return None
    with torch.no_grad():
        X, U, Om, r = (torch.from_numpy(v).cuda() for v in particles(c, seed))
        n = len(r)
        F = body_force(c)
        none = torch.zeros((n, 3), dtype=torch.float64, device="cuda")
        if c["kind"] == "dem":
            law = Contacts(c, X, r)
            for _ in range(c["substeps"] * c["steps"]):
                X, U, Om = law.step(X, U, Om, none, none)
            return dict(X=X, U=U, Om=Om)
        fl = Fluid(c)
        fl.count = n
        if c["kind"] == "buffers":
            scale = 4096.0 if c["storage"] == "f16" else 1.0
            g = (flow(c, seed) * scale).to(TYPES[c["storage"]]).double() / scale
            g, Ft = fl.collide(fl.pull(g), F, fl.shells(X, r), U, Om)
            return dict(f=g * scale, F=Ft[0], T=Ft[1])
        g = fl.unpull(flow(c, seed))
        if c["kind"] == "adjoint":
            return gradient(fl, c, g, X, r)
        law = Contacts(c, X, r) if c["kind"] == "coupled" else None
        shell = fl.shells(X, r) if n else None
        moving = c["kind"] in ("coupled", "driven", "buffers")
        FT = []
        for k in range(c["steps"]):
            if k and moving:
                shell = fl.shells(X + k * U if c["kind"] == "driven" else X, r)
            g, Ft = fl.collide(fl.pull(g), F, shell, U if moving else None, Om if moving else None)
            FT.append(Ft or (none, none))
            if law:
                for _ in range(c["substeps"]):
                    X, U, Om = law.step(X, U, Om, *Ft)
        drho, _, u = fl.moments(fl.pull(g), F)
        out = dict(F=FT[-1][0], T=FT[-1][1], rho=1 + drho, u=torch.stack([v.expand(drho.shape) for v in u], -1))
        if c["kind"] == "driven":
            out["F"], out["T"] = (torch.stack([v[k] for v in FT]) for k in (0, 1))
        if law:
            out.update(X=X, U=U, Om=Om)
        return out


def gradient(fl, c, g, X, r):
    """J, dJ/dX and dJ/dF by automatic differentiation of the steps."""
    from torch.utils.checkpoint import checkpoint

    def one(g, Xd, Fd):
        out, Ft = fl.collide(fl.pull(g), Fd, fl.shells(X, r, Xd))
        return out, Ft[0][:, 0].sum()

    with torch.enable_grad():
        Xd = X.clone().requires_grad_()
        Fd = torch.tensor(body_force(c), dtype=torch.float64, device="cuda", requires_grad=True)
        J = 0.0
        for _ in range(c["steps"]):
            g, d = checkpoint(one, g, Xd, Fd, use_reentrant=False)
            J = J + d / c["steps"]
        J.backward()
    return dict(J=J.detach().reshape(1), dX=Xd.grad, dF=Fd.grad)
