"""What a program that uses this library has it do, as cases that can be timed.

A pass is what such a program does between two snapshots: a number of
dust_step calls on grains that stay in the library, then the read-back of the
grains, the gas and the deposit into the program's own device arrays.  Other
passes are the exchange of every grain with a host code each step, the step
on caller-owned arrays (dust_step_noalloc), the batched step of many small
boxes, and the dust density diagnostic.

Inputs are drawn on the GPU from the seed, with the distributions of
paper_1908_10793_gb300/inputs.py.  Grains of the disks start a few zones away
from the open radial boundary, so none leaves in the compared passes (removed
grains are read back in no particular order).

exact() restates the step in 64-bit torch: the deposit and the gas of every
kind of pass, and the grains where a pass returns them in the caller's order.
"""
import math

import numpy as np
import torch

from paper_1908_10793_gb300 import dust as D
from paper_1908_10793_gb300 import inputs as I

DEV = "cuda"
WEIGHTS = {"cic": I.CIC, "tsc": I.TSC, "volume": I.VOLUME}


def listed():
    def c(name, kind, n, grains, steps, **kw):
        d = dict(name=name, kind=kind, geom="shear", n0=n[0], n1=n[1], n2=n[2], grains=grains, steps=steps,
                 precision="mixed", weight="tsc", feedback=True, predictor=False)
        d.update(kw)
        return d

    return [
        # the deceleration setup on a 64^2 periodic box: the smallest run,
        # where a step is a handful of short launches
        c("box_64x64", "evolve", (64, 64, 1), 16384, 50, geom="box"),
        # a shearing box whose sides are no multiple of the tile, six grains
        # per zone: the sizes of a resolution study's first runs
        c("shear_50x37x29", "evolve", (50, 37, 29), 321900, 20),
        # the benchmark's shearing box, eight grains per zone
        c("shear_128", "evolve", (128, 128, 128), 16777216, 10),
        # the global cylindrical disk: four species, two grains per zone,
        # log-spaced radius, feedback; the largest run
        c("cyl_disk", "evolve", (384, 1024, 64), 50_000_000, 4, geom="cyl"),
        # the global spherical disk: a stopping time per grain over five
        # decades, gas held fixed
        c("sph_disk", "evolve", (256, 128, 512), 33_000_000, 4, geom="sph", feedback=False),
        # the disk with the gas half-step predictor
        c("cyl_predictor", "evolve", (192, 512, 32), 6_250_000, 4, geom="cyl", predictor=True),
        # the disk with the traditional volume weighting, for comparison runs
        c("cyl_volume", "evolve", (192, 512, 32), 6_250_000, 4, geom="cyl", weight="volume"),
        # a double-precision run, as a check of a mixed-precision one
        c("shear_fp64_64", "evolve", (64, 64, 64), 2097152, 4, precision="fp64"),
        # a parameter study: 64 axisymmetric boxes of 32^2 to 512^2 zones and
        # 1 to 16 grains per zone in one batch
        c("si_batch_64", "batch", (512, 1, 512), 0, 10, instances=64),
        # a host gas code that keeps the grains itself: load, step and read
        # back through pinned memory every step
        c("host_exchange_96", "host", (96, 96, 96), 7077888, 1),
        # a host code that owns the device memory: the allocation-free step
        # in double precision, grains in no order
        c("noalloc_64", "noalloc", (64, 64, 64), 2097152, 1, precision="fp64"),
        # the dust density between steps
        c("mass_disk", "mass", (192, 512, 32), 6_250_000, 1, geom="cyl"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["evolve"] * 6 + ["batch", "host", "noalloc", "mass"])
    d = dict(kind=kind, geom="shear", n0=1, n1=1, n2=1, grains=0, steps=1, precision="mixed", weight="tsc",
             feedback=True, predictor=False)
    if kind == "batch":
        d["instances"] = rng.randint(3, 64)
        d["n0"] = d["n2"] = 512
        d["steps"] = rng.randint(2, 12)
        return d
    if kind == "evolve":
        d["geom"] = rng.choice(["box", "shear", "shear", "cyl", "cyl", "sph"])
        d["precision"] = rng.choice(["mixed"] * 5 + ["fp64"])
        d["predictor"] = rng.random() < 0.15
        d["steps"] = rng.randint(2, 8)
    elif kind in ("noalloc", "mass"):
        d["geom"] = rng.choice(["shear", "cyl", "sph"])
        d["precision"] = "fp64" if kind == "noalloc" else "mixed"
    fp64 = d["precision"] == "fp64"
    d["weight"] = rng.choice(["tsc"] * 4 + ["cic"] + (["volume"] if d["geom"] in ("cyl", "sph") else []))
    d["feedback"] = d["geom"] != "sph" and rng.random() < 0.8
    if d["geom"] == "box":
        d["n0"], d["n1"] = _log(rng, 17, 700), _log(rng, 17, 700)
    elif d["geom"] == "shear":
        big = 70 if fp64 or kind == "host" else 130
        d["n0"], d["n1"], d["n2"] = (_log(rng, 14, big) for _ in range(3))
    elif d["geom"] == "cyl":
        s = 0.4 if fp64 else 1.0
        d["n0"], d["n1"], d["n2"] = _log(rng, 24, 300 * s), _log(rng, 32, 700 * s), _log(rng, 8, 60 * s)
    else:
        s = 0.4 if fp64 else 1.0
        d["n0"], d["n1"], d["n2"] = _log(rng, 16, 200 * s), _log(rng, 16, 100 * s), _log(rng, 16, 400 * s)
    zones = d["n0"] * d["n1"] * d["n2"]
    ppz = math.exp(rng.uniform(math.log(1.2), math.log(14.0)))
    d["grains"] = max(1000, min(int(zones * ppz), 4_000_000 if fp64 else 30_000_000)) | 1
    return d


# ------------------------------------------------------------ the setups --

def _edges(lo, hi, n, log=False):
    t = np.arange(n + 1, dtype=np.float64) / n
    e = lo * (hi / lo) ** t if log else lo + (hi - lo) * t
    e[0], e[-1] = lo, hi
    return e


def _workload(case):
    """The library's descriptors of a case (no grains, no gas)."""
    geom, n, N = case["geom"], (case["n0"], case["n1"], case["n2"]), max(case["grains"], 1)
    kw = dict(rho=None, vgas=[], q=[], v=[], steps=case["steps"], feedback=int(case["feedback"]),
              weight=WEIGHTS[case["weight"]], name=geom)
    if geom == "box":
        return I.Workload(geom=I.CARTESIAN, edges=[_edges(0.0, 1.0, n[0]), _edges(0.0, 1.0, n[1]), np.array([0.0, 1.0])],
                          bc=[I.PERIODIC] * 3, species_mass=[1.0 / N], species_tau_mode=[I.TAU_CONST],
                          species_tau=[0.1], dt=min(0.01, 0.64 / max(n)), **kw)
    if geom == "shear":
        L = 0.2
        return I.Workload(geom=I.SHEARING_BOX, edges=[_edges(-0.5 * L, 0.5 * L, m) for m in n], bc=[I.PERIODIC] * 3,
                          species_mass=[0.02 * L ** 3 / N], species_tau_mode=[I.TAU_STOKES], species_tau=[0.1],
                          dt=5e-3, fargo=1, omega=1.0, qshear=1.5, **kw)
    if geom == "cyl":
        mass = 0.01 * 2.1 * 2.0 * np.pi * 0.3 / N
        return I.Workload(geom=I.CYLINDRICAL, edges=[_edges(0.4, 2.5, n[0], True), _edges(0.0, 2.0 * np.pi, n[1]),
                                                     _edges(-0.15, 0.15, n[2])],
                          bc=[I.OUTFLOW, I.PERIODIC, I.PERIODIC], species_mass=[mass] * 4,
                          species_tau_mode=[I.TAU_STOKES] * 4, species_tau=[0.01, 0.1, 1.0, 10.0], dt=1e-3, gm=1.0, **kw)
    return I.Workload(geom=I.SPHERICAL, edges=[_edges(0.5, 3.0, n[0], True),
                                               _edges(0.5 * np.pi - 0.3, 0.5 * np.pi + 0.3, n[1]),
                                               _edges(0.0, 2.0 * np.pi, n[2])],
                      bc=[I.OUTFLOW, I.OUTFLOW, I.PERIODIC], species_mass=[1e-3 / N], species_tau_mode=[I.TAU_STOKES],
                      species_tau=[1.0], dt=2e-3, gm=1.0, **kw)


def _centres(w):
    """Zone-centre coordinates on the GPU, in storage order."""
    c = [torch.tensor(0.5 * (e[1:] + e[:-1]), device=DEV) for e in w.edges]
    z, y, x = torch.meshgrid(c[2], c[1], c[0], indexing="ij")
    return x.reshape(-1), y.reshape(-1), z.reshape(-1)


def _inside(x, lo, hi):
    """Coordinates as a program hands them over: inside the half-open range."""
    return x.clamp_(min=lo, max=float(np.nextafter(hi, lo)))


def _data(case, seed, w):
    """Grains and gas of a case: (q, v, species, param, rho, vgas)."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    N, nc = case["grains"], w.ncell

    def uni(lo, hi):
        return _inside(torch.rand(N, generator=g, device=DEV, dtype=torch.float64).mul_(hi - lo).add_(lo), lo, hi)

    def normal(m):
        return torch.randn(m, generator=g, device=DEV, dtype=torch.float64)

    lo, hi = [e[0] for e in w.edges], [e[-1] for e in w.edges]
    one = torch.ones(nc, device=DEV, dtype=torch.float64)
    if case["geom"] == "box":
        q = [uni(lo[0], hi[0]), uni(lo[1], hi[1]), torch.full((N,), 0.5, device=DEV, dtype=torch.float64)]
        v = [normal(N), normal(N), torch.zeros(N, device=DEV, dtype=torch.float64)]
        return q, v, None, None, one, [one * 0.3, one * -0.2, one * 0.0]
    if case["geom"] == "shear":
        if case["kind"] in ("host", "noalloc"):
            q = [uni(lo[d], hi[d]) for d in range(3)]
        else:
            q = _zone_by_zone(g, w, N)
        v = [normal(N) * 1e-3 for _ in range(3)]
        return q, v, None, None, one, [normal(nc) * 1e-3 for _ in range(3)]
    x, y, _ = _centres(w)
    if case["geom"] == "cyl":
        R = uni(lo[0] * 1.03, hi[0] * 0.97)
        q = [R, uni(lo[1], hi[1]), uni(lo[2], hi[2])]
        v = [torch.zeros_like(R), R ** -0.5, torch.zeros_like(R)]
        species = torch.randint(0, 4, (N,), generator=g, device=DEV, dtype=torch.uint8)
        vk = x ** -0.5
        return q, v, species, None, 1.0 / x, [1e-3 * vk * normal(nc), vk * (1.0 + 1e-3 * normal(nc)), 1e-3 * vk * normal(nc)]
    a, b = (lo[0] * 1.03) ** 1.5, (hi[0] * 0.97) ** 1.5
    r = uni(a, b) ** (2.0 / 3.0)
    th = 0.5 * np.pi - torch.atan((0.05 * normal(N)).clamp_(-0.27, 0.27))
    q = [r, th, uni(lo[2], hi[2])]
    v = [torch.zeros_like(r), torch.zeros_like(r), (r * torch.sin(th)) ** -0.5]
    param = 10.0 ** uni(-4.0, 1.0)
    vk = (x * torch.sin(y)) ** -0.5
    rho = x ** -1.5 * torch.exp(-(1.0 / torch.tan(y)) ** 2 / (2.0 * 0.05 ** 2))
    return q, v, None, param, rho, [1e-3 * vk * normal(nc), 1e-3 * vk * normal(nc), vk * (1.0 + 1e-3 * normal(nc))]


def _zone_by_zone(g, w, N):
    """N grains spread evenly over the zones, uniform inside each, in zone
    order, as an initial condition is laid out."""
    z = torch.arange(N, device=DEV) * w.ncell // N
    idx = [z % w.n[0], (z // w.n[0]) % w.n[1], z // (w.n[0] * w.n[1])]
    q = []
    for d in range(3):
        e = torch.tensor(w.edges[d], device=DEV)
        f = torch.rand(N, generator=g, device=DEV, dtype=torch.float64)
        q.append(_inside(e[idx[d]] + (e[idx[d] + 1] - e[idx[d]]) * f, w.edges[d][0], w.edges[d][-1]))
    return q


def _instances(case, seed):
    """(workload, data) of each box of the batch: the grids, Stokes numbers and
    dust-to-gas ratios of inputs.si2d_instance, equilibrium drift, noise in the
    gas."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    got = []
    for k in range(case["instances"]):
        side, ppc, st, eps = 32 * 2 ** (k % 5), 1 + k % 16, (0.01, 0.1, 1.0)[k % 3], (0.01, 0.02, 0.1)[(k // 3) % 3]
        nc, L = side * side, 0.2
        N = nc * ppc
        w = I.Workload(name="si", geom=I.SHEARING_BOX, edges=[_edges(-0.1, 0.1, side), np.array([-0.1, 0.1]), _edges(-0.1, 0.1, side)],
                       bc=[I.PERIODIC] * 3, weight=I.TSC, species_mass=[eps * (L / side) ** 2 * L / ppc],
                       species_tau_mode=[I.TAU_STOKES], species_tau=[st], rho=None, vgas=[], q=[], v=[], dt=5e-3,
                       steps=case["steps"], feedback=1, fargo=1, omega=1.0, qshear=1.5)
        f, drift = (1.0 + eps) ** 2 + st ** 2, 0.05

        def const(m, x):
            return torch.full((m,), x, device=DEV, dtype=torch.float64)

        q = _zone_by_zone(g, w, N)
        v = [const(N, -2.0 * st / f * drift), const(N, -(1.0 - st ** 2 / f) / (1.0 + eps) * drift), const(N, 0.0)]
        mean = [2.0 * eps * st / f * drift, -(1.0 + eps * st ** 2 / f) / (1.0 + eps) * drift, 0.0]
        vgas = [m + 1e-3 * torch.randn(nc, generator=g, device=DEV, dtype=torch.float64) for m in mean]
        got.append((w, (q, v, None, None, const(nc, 1.0), vgas)))
    return got


class _State:
    """What a program holds: contexts, its own device arrays, a batch."""
    batch = None

    def __del__(self):
        try:
            if self.batch is not None:
                D.dust_batch_destroy(self.batch)
                self.batch = None
            for c in self.ctx:
                c.close()
        except Exception:
            pass


def _context(case, w, **kw):
    return D.Context(w, precision=D.DUST_FP64 if case["precision"] == "fp64" else D.DUST_MIXED,
                     gas_predictor=int(case["predictor"]), **kw)


def _outputs(n, nc, velocity, make=None):
    make = make or (lambda m, t: torch.empty(m, device=DEV, dtype=t))
    return dict(q=[make(n, torch.float64) for _ in range(3)], v=[make(n, velocity) for _ in range(3)],
                ids=make(n, torch.int64), dep=make((nc, 4), torch.float64), gas=[make(nc, torch.float64) for _ in range(4)])


def prepare(case, seed):
    s = _State()
    s.case, s.ctx = case, []
    kind = case["kind"]
    if kind == "batch":
        ws = _instances(case, seed)
        torch.cuda.synchronize()  # the library reads these arrays on its own streams
        s.n, s.nc, s.dt = [len(x[0][0]) for _, x in ws], [w.ncell for w, _ in ws], [w.dt for w, _ in ws]
        for w, (q, v, species, param, rho, vgas) in ws:
            c = _context(case, w)
            s.ctx.append(c)
            c.set_gas(rho, vgas)
            c.load(q, v, species, param)
        s.batch = D.dust_batch_create([c.handle for c in s.ctx])
        s.out = _outputs(sum(s.n), sum(s.nc), torch.float32)
        return s
    w = _workload(case)
    q, v, species, param, rho, vgas = _data(case, seed, w)
    torch.cuda.synchronize()  # the library reads these arrays on its own stream
    s.w, s.n, s.nc = w, case["grains"], w.ncell
    if kind == "noalloc":
        s.desc = D.make_descriptors(w, precision=D.DUST_FP64)
        gas = [rho] + list(_momentum(w, _centres(w), vgas))
        s.q, s.p = [x.clone() for x in q], [x.contiguous() for x in _momentum(w, q, v)]
        s.gas, s.species, s.param, s.t = torch.stack(gas, 1).contiguous(), species, param, 0.0
        s.dep = torch.empty((s.nc, 4), device=DEV, dtype=torch.int64)
        s.status = torch.zeros(4, device=DEV, dtype=torch.int32)
        return s
    if kind == "host":
        def pin(x):
            return torch.empty(x.shape, dtype=x.dtype, pin_memory=True).copy_(x)

        s.q, s.v = [pin(x) for x in q], [pin(x.float()) for x in v]
        s.gas = [pin(x) for x in [rho] + vgas]
        s.species, s.param = (None if x is None else pin(x) for x in (species, param))
        s.ctx.append(_context(case, w, host_io_async=1))
        s.out = _outputs(s.n, s.nc, torch.float32, lambda m, t: torch.empty(m, dtype=t, pin_memory=True))
        return s
    s.ctx.append(_context(case, w))
    s.ctx[0].set_gas(rho, vgas)
    s.ctx[0].load(q, v, species, param)
    if kind == "mass":  # called between steps: the grains are in zone order
        s.ctx[0].step(w.dt)
        s.ctx[0].sync(check=False)
        s.mass = torch.empty(s.nc, device=DEV, dtype=torch.float64)
    else:
        s.out = _outputs(s.n, s.nc, torch.float64 if case["precision"] == "fp64" else torch.float32)
    return s


def _read(ctx, n, q, v, ids, dep, gas):
    """The snapshot: grains, deposit of the last step, gas."""
    get = D.dust_get_particles_v32 if v[0].dtype == torch.float32 else D.dust_get_particles
    get(ctx, n, q[0], q[1], q[2], v[0], v[1], v[2], ids)
    D.dust_get_deposit(ctx, as_double=dep)
    if gas is not None:
        D.dust_get_gas(ctx, gas[0], gas[1], gas[2], gas[3])


def run(s):
    case, kind = s.case, s.case["kind"]
    if kind == "batch":
        D.dust_batch_step(s.batch, s.dt, case["steps"])
        o, a, b = s.out, 0, 0
        for c, n, nc in zip(s.ctx, s.n, s.nc):
            _read(c.handle, n, [x[a:a + n] for x in o["q"]], [x[a:a + n] for x in o["v"]], o["ids"][a:a + n],
                  o["dep"][b:b + nc], [x[b:b + nc] for x in o["gas"]])
            a, b = a + n, b + nc
        return o
    if kind == "noalloc":
        geo, grid, sp, opt, _ = s.desc
        D.dust_step_noalloc(geo, grid, sp, s.w.weight, 0.0, s.t, s.w.dt, s.q, s.p, s.gas, s.dep, species_idx=s.species,
                            param=s.param, status_out=s.status, stream=torch.cuda.current_stream().cuda_stream)
        s.t += s.w.dt
        return dict(q=s.q, p=s.p, dep=s.dep.double(), status=s.status)
    h = s.ctx[0].handle
    if kind == "mass":
        D.dust_get_mass_deposit(h, as_double=s.mass)
        return s.mass
    if kind == "host":
        D.dust_load_particles_v32(h, s.q[0], s.q[1], s.q[2], s.v[0], s.v[1], s.v[2], s.species, s.param)
        D.dust_set_gas(h, s.gas[0], s.gas[1], s.gas[2], s.gas[3])
        D.dust_step(h, s.w.dt)
        _read(h, s.n, s.out["q"], s.out["v"], s.out["ids"], s.out["dep"], None)
        D.dust_sync(h, check=False)
        return {k: s.out[k] for k in ("q", "v", "ids", "dep")}
    for _ in range(case["steps"]):
        D.dust_step(h, s.w.dt)
    _read(h, s.n, s.out["q"], s.out["v"], s.out["ids"], s.out["dep"], s.out["gas"])
    return s.out


def work(case):
    """Per step: a grain's 36 (mixed) or 48 (double) bytes of coordinates and
    momenta read and written, its species byte or stopping time read, a zone's
    gas read (and written with feedback) and deposit written.  Per pass: the
    snapshot's columns read and written.  Operations: the 27-node gather and
    deposit of four channels and about 150 for weights, kick and drifts."""
    if case["kind"] == "batch":
        sides = [32 * 2 ** (k % 5) for k in range(case["instances"])]
        n = sum(m * m * (1 + k % 16) for k, m in enumerate(sides))
        nc, nodes = sum(m * m for m in sides), 9
    else:
        n, nc = case["grains"], case["n0"] * case["n1"] * case["n2"]
        nodes = 9 if 1 in (case["n0"], case["n1"], case["n2"]) else 27
    fp64 = case["precision"] == "fp64"
    state, gas = (48, 32) if fp64 else (36, 16)
    extra = {"cyl": 1, "sph": 8 if fp64 else 4}.get(case["geom"], 0)
    fb = gas if case["feedback"] else 0
    flops = n * (16 * nodes + 150)
    if case["kind"] == "mass":
        return {"bytes": n * (24 + extra) + nc * 8, "flops": n * (4 * nodes + 30)}
    if case["kind"] == "host":
        return {"bytes": n * (36 + extra + 44) + nc * (32 + 32), "flops": flops}
    if case["kind"] == "noalloc":
        return {"bytes": n * (2 * state + (8 if case["geom"] == "sph" else extra)) + nc * (gas + 32), "flops": flops}
    pred = n * (state + extra) + nc * (gas + 32) if case["predictor"] else 0
    step = n * (2 * state + extra) + nc * (gas + fb + 32) + pred
    snap = n * (state + 4 + 24 + (24 if fp64 else 12) + 8) + nc * (64 + gas + 32)
    return {"bytes": case["steps"] * step + snap, "flops": case["steps"] * flops * (2 if case["predictor"] else 1)}


# -------------------------------------------------- the step in 64 bits ---

def _momentum(w, q, v, inverse=False):
    """Physical velocity to the momentum-like variables at q, or back."""
    if w.geom == I.CYLINDRICAL:
        f = [None, q[0], None]
    elif w.geom == I.SPHERICAL:
        f = [None, q[0], q[0] * torch.sin(q[1])]
    else:
        f = [None, None, None]
    return [x if m is None else (x / m if inverse else x * m) for x, m in zip(v, f)]


def _node(i, n, periodic):
    return i % n if periodic else i.clamp(0, n - 1)


def _weights(w, d, x):
    """Host zone of x in direction d and the three weights (Sec. 3.4, App. C)."""
    n = w.n[d]
    if n == 1:
        return torch.zeros_like(x, dtype=torch.int64), None
    e = torch.tensor(w.edges[d], device=DEV)
    i = (torch.searchsorted(e, x, right=True) - 1).clamp_(0, n - 1)
    c, dx = 0.5 * (e[i] + e[i + 1]), e[i + 1] - e[i]
    u = (x - c) / dx
    up, dn = u.clamp(min=0.0), (-u).clamp(min=0.0)
    radial = d == 0 and w.geom in (I.CYLINDRICAL, I.SPHERICAL)
    polar = d == 1 and w.geom == I.SPHERICAL
    if w.weight == I.VOLUME and (radial or polar):
        cc = torch.cat([e[:1] - 0.5 * (e[1] - e[0]), 0.5 * (e[1:] + e[:-1]), e[-1:] + 0.5 * (e[-1] - e[-2])])

        def shell(a, b):  # volume between a and b
            if polar:
                return 2.0 * torch.sin(0.5 * (a + b)) * torch.sin(0.5 * (b - a))
            return (b - a) * (b + a) if w.geom == I.CYLINDRICAL else (b - a) * (a * a + a * b + b * b)

        h = torch.where(x >= c, shell(c, x) / shell(c, cc[i + 2]), 0.0)
        lo = torch.where(x < c, shell(x, c) / shell(cc[i], c), 0.0)
        return i, (lo, 1.0 - lo - h, h)
    if w.weight != I.TSC and not radial and not polar:
        return i, (dn, 1.0 - dn - up, up)
    if not radial and not polar:
        return i, (0.5 * (0.5 - u) ** 2, 0.75 - u * u, 0.5 * (0.5 + u) ** 2)
    # the shape times the direction's measure, integrated over each zone of
    # width dx: Gauss points on the pieces of the spline (the measure is a
    # polynomial of degree two, or a sine over one zone)
    t, g = np.polynomial.legendre.leggauss(8)

    def measure(y):
        return torch.sin(y) if polar else (y if w.geom == I.CYLINDRICAL else y * y)

    def integral(a, b, shape):  # over offsets s from the grain, in zone widths
        m, r, s = 0.5 * (a + b), 0.5 * (b - a), 0.0
        for tk, gk in zip(t, g):
            z = m + r * tk
            s = s + gk * shape(z) * measure(x + z * dx)
        return s * r

    if w.weight == I.TSC:  # triangle of half width one
        def shape(z):
            return 1.0 - z.abs()

        lo = integral(torch.full_like(u, -1.0), -0.5 - u, shape)
        h = integral(0.5 - u, torch.full_like(u, 1.0), shape)
        zero = torch.zeros_like(u)
        mid = integral(-0.5 - u, zero, shape) + integral(zero, 0.5 - u, shape)
    else:  # top hat of one zone
        half, flat = torch.full_like(u, 0.5), torch.ones_like
        lo = integral(-half, torch.maximum(-half, -0.5 - u), flat)
        h = integral(torch.minimum(half, 0.5 - u), half, flat)
        mid = integral(torch.maximum(-half, -0.5 - u), torch.minimum(half, 0.5 - u), flat)
    s = lo + mid + h
    return i, (lo / s, mid / s, h / s)


def _stencil(w, q):
    z = [_weights(w, d, q[d]) for d in range(3)]
    rng = [range(3) if w.n[d] > 1 else (1,) for d in range(3)]
    for c in rng[2]:
        for b in rng[1]:
            for a in rng[0]:
                k = [_node(z[d][0] + o - 1, w.n[d], w.bc[d] == I.PERIODIC) for d, o in enumerate((a, b, c))]
                W = None
                for d, o in enumerate((a, b, c)):
                    if z[d][1] is not None:
                        W = z[d][1][o] if W is None else W * z[d][1][o]
                yield (a, b, c), k[0] + w.n[0] * (k[1] + w.n[1] * k[2]), W


def _gather(w, q, fields):
    out = [torch.zeros_like(q[0]) for _ in fields]
    for _, k, W in _stencil(w, q):
        for o, f in zip(out, fields):
            o.addcmul_(W, f[k])
    return out


def _deposit(w, q, values, out):
    """out[:, c] += sum of W * values[c]: zone sums from differences of the
    running sum over grains in zone order, then shifted to the node."""
    host = [_weights(w, d, q[d])[0] for d in range(3)]
    zone = host[0] + w.n[0] * (host[1] + w.n[1] * host[2])
    zone, order = torch.sort(zone)
    ends = torch.searchsorted(zone, torch.arange(w.ncell + 1, device=DEV))
    idx = torch.arange(w.ncell, device=DEV)
    hz = [idx % w.n[0], (idx // w.n[0]) % w.n[1], idx // (w.n[0] * w.n[1])]
    qs, vs = [x[order] for x in q], [x[order] for x in values]
    for o, _, W in _stencil(w, qs):
        k = [_node(hz[d] + o[d] - 1, w.n[d], w.bc[d] == I.PERIODIC) for d in range(3)]
        k = k[0] + w.n[0] * (k[1] + w.n[1] * k[2])
        for c, x in enumerate(vs):
            run_ = torch.zeros(len(zone) + 1, device=DEV, dtype=torch.float64)
            torch.cumsum(W * x if W is not None else x, 0, out=run_[1:])
            out[:, c].index_add_(0, k, run_[ends[1:]] - run_[ends[:-1]])


def _drift(w, q, qm, p, h, second):
    q = list(q)
    q[0] = q[0] + h * p[0]
    m = qm if second else q
    if w.geom == I.CYLINDRICAL:
        q[1] = q[1] + h * p[1] / m[0] ** 2
        q[2] = q[2] + h * p[2]
    elif w.geom == I.SPHERICAL:
        q[1] = q[1] + h * p[1] / m[0] ** 2
        q[2] = q[2] + h * p[2] / (m[0] * torch.sin((qm if second else q)[1])) ** 2
    elif w.geom == I.SHEARING_BOX:
        q[1] = q[1] + h * (p[1] - w.qshear * w.omega * m[0])
        q[2] = q[2] + h * p[2]
    else:
        q[1], q[2] = q[1] + h * p[1], q[2] + h * p[2]
    return q


def _wrap(w, q, t):
    if w.geom == I.SHEARING_BOX:
        L, Ly = w.edges[0][-1] - w.edges[0][0], w.edges[1][-1] - w.edges[1][0]
        s = math.fmod(w.qshear * w.omega * L * t, Ly)
        q[1] = q[1] + s * ((q[0] >= w.edges[0][-1]).double() - (q[0] < w.edges[0][0]).double())
    for d in range(3):
        if w.bc[d] == I.PERIODIC:
            lo, hi = w.edges[d][0], w.edges[d][-1]
            for _ in range(2):
                q[d] = torch.where(q[d] >= hi, q[d] - (hi - lo), torch.where(q[d] < lo, q[d] + (hi - lo), q[d]))
    return q


def _volume(w):
    e = [torch.tensor(x, device=DEV) for x in w.edges]
    v = [x[1:] - x[:-1] for x in e]
    if w.geom == I.CYLINDRICAL:
        v[0] = 0.5 * (e[0][1:] ** 2 - e[0][:-1] ** 2)
    if w.geom == I.SPHERICAL:
        v[0], v[1] = (e[0][1:] ** 3 - e[0][:-1] ** 3) / 3.0, torch.cos(e[1][:-1]) - torch.cos(e[1][1:])
    return (v[2][:, None, None] * v[1][None, :, None] * v[0][None, None, :]).reshape(-1)


def _tau(w, q, species, param):
    St = param if param is not None else torch.tensor(w.species_tau, device=DEV, dtype=torch.float64)[
        species.long() if species is not None else torch.zeros_like(q[0], dtype=torch.int64)]
    if w.species_tau_mode[0] == I.TAU_CONST:
        return St
    if w.geom == I.SHEARING_BOX:
        return St / w.omega
    R = q[0] * torch.sin(q[1]) if w.geom == I.SPHERICAL else q[0]
    return St * torch.sqrt(R ** 3 / w.gm)


def _kick(w, q, p, vg, tau, dt):
    """New p, non-frictional acceleration, dH/dp at the half step."""
    x = dt / tau
    E, cg = torch.exp(-x), -torch.expm1(-x)
    h1 = cg * tau
    z = torch.zeros_like(p[0])
    if w.geom == I.SHEARING_BOX:
        Om, qs = w.omega, w.qshear
        r0 = E * p[0] + h1 * Om * p[1] + cg * vg[0]
        r1 = E * p[1] + h1 * 0.5 * (qs - 2.0) * Om * p[0] + cg * vg[1]
        o1, o2 = Om * h1, Om * h1 * (1.0 - 0.5 * qs)
        det = 1.0 + o1 * o2
        n = [(r0 + o1 * r1) / det, (r1 - o2 * r0) / det, E * p[2] + cg * vg[2]]
        dH = [0.5 * (a + b) for a, b in zip(p, n)]
        return n, [2.0 * Om * dH[1], (qs - 2.0) * Om * dH[0], z], dH
    if w.geom == I.CYLINDRICAL:
        R = q[0]
        n1 = E * p[1] + cg * vg[1]
        a0 = 0.5 * (p[1] ** 2 + n1 ** 2) / R ** 3 - w.gm / R ** 2
        n = [E * p[0] + h1 * a0 + cg * vg[0], n1, E * p[2] + cg * vg[2]]
        dH = [0.5 * (p[0] + n[0]), 0.5 * (p[1] + n[1]) / R ** 2, 0.5 * (p[2] + n[2])]
        return n, [a0, z, z], dH
    if w.geom == I.SPHERICAL:
        r, st, ct = q[0], torch.sin(q[1]), torch.cos(q[1])
        n2 = E * p[2] + cg * vg[2]
        l2 = 0.5 * (p[2] ** 2 + n2 ** 2)
        a1 = l2 * ct / (r ** 2 * st ** 3)
        n1 = E * p[1] + h1 * a1 + cg * vg[1]
        a0 = (0.5 * (p[1] ** 2 + n1 ** 2) + l2 / st ** 2) / r ** 3 - w.gm / r ** 2
        n = [E * p[0] + h1 * a0 + cg * vg[0], n1, n2]
        dH = [0.5 * (p[0] + n[0]), 0.5 * (p[1] + n[1]) / r ** 2, 0.5 * (p[2] + n[2]) / (r * st) ** 2]
        return n, [a0, a1, z], dH
    n = [E * a + cg * b for a, b in zip(p, vg)]
    return n, [z, z, z], [0.5 * (a + b) for a, b in zip(p, n)]


def _steps64(w, data, steps, feedback, predictor):
    """q, p, deposit of the last step, gas momentum after `steps` steps."""
    q, v, species, param, rho, vgas = data
    p = _momentum(w, q, v)
    gas = [x.clone() for x in _momentum(w, _centres(w), vgas)]
    dV, dt, t, chunk = _volume(w), w.dt, 0.0, 6_000_000
    m = w.species_mass[0]
    parts = [slice(a, min(a + chunk, len(q[0]))) for a in range(0, len(q[0]), chunk)]
    q, p = [x.clone() for x in q], [x.clone() for x in p]
    dep = None

    def of(x, sl):
        return None if x is None else x[sl]

    for _ in range(steps):
        half = gas
        if predictor:
            imp = torch.zeros(w.ncell, 3, device=DEV, dtype=torch.float64)
            for sl in parts:
                a, b = [x[sl] for x in q], [x[sl] for x in p]
                vg = _gather(w, a, gas)
                tau = _tau(w, a, of(species, sl), of(param, sl)).clamp(min=abs(dt))
                _deposit(w, a, [0.5 * dt * m * (y - z) / tau for y, z in zip(b, vg)], imp)
            half = [g + imp[:, c] / (rho * dV) for c, g in enumerate(gas)]
        dep = torch.zeros(w.ncell, 4, device=DEV, dtype=torch.float64)
        for sl in parts:
            b = [x[sl] for x in p]
            a = _wrap(w, _drift(w, [x[sl] for x in q], None, b, 0.5 * dt, False), t + 0.5 * dt)
            vg = _gather(w, a, half)
            n, acc, dH = _kick(w, a, b, vg, _tau(w, a, of(species, sl), of(param, sl)), dt)
            dp = [-m * ((y - z) - dt * f) for y, z, f in zip(n, b, acc)]
            _deposit(w, a, dp + [sum(x * y for x, y in zip(dp, dH))], dep)
            a = _wrap(w, _drift(w, a, a, n, 0.5 * dt, True), t + dt)
            for d in range(3):
                q[d][sl], p[d][sl] = a[d], n[d]
        if feedback:
            gas = [g + dep[:, c] / (rho * dV) for c, g in enumerate(gas)]
        t += dt
    return q, p, dep, gas


def exact(case, seed):
    """Grains read back in the library's storage order have no value here (the
    order depends on the library's own rounding of zone edges)."""
    none3 = [None, None, None]
    if case["kind"] == "batch":
        if case["instances"] * case["steps"] > 700:
            return None
        deps, gases = [], []
        for w, data in _instances(case, seed):
            _, _, dep, gas = _steps64(w, data, case["steps"], True, False)
            deps.append(dep)
            gases.append([data[4]] + gas)
        return dict(q=none3, v=none3, ids=None, dep=torch.cat(deps), gas=[torch.cat(x) for x in zip(*gases)])
    w = _workload(case)
    data = _data(case, seed, w)
    if case["grains"] * case["steps"] > 210_000_000:
        return None
    if case["kind"] == "mass":
        q, _, _, _ = _steps64(w, data, 1, case["feedback"], False)
        out = torch.zeros(w.ncell, 1, device=DEV, dtype=torch.float64)
        for a in range(0, len(q[0]), 6_000_000):
            part = [x[a:a + 6_000_000] for x in q]
            _deposit(w, part, [torch.full_like(part[0], w.species_mass[0])], out)
        return out[:, 0]
    q, p, dep, gas = _steps64(w, data, case["steps"], case["feedback"] and case["kind"] != "noalloc", case["predictor"])
    if case["kind"] == "noalloc":
        quantum = math.ldexp(w.species_mass[0], -44)
        return dict(q=q, p=p, dep=dep / quantum, status=None)
    if case["kind"] == "host":
        return dict(q=none3, v=none3, ids=None, dep=dep)
    return dict(q=none3, v=none3, ids=None, dep=dep, gas=[data[4]] + _momentum(w, _centres(w), gas, inverse=True))
