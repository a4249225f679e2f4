"""The work a user of the library has it do, as timed cases.

Every case goes through the public binding (paper_1101_0809_gb300.pic) or the
differentiable run (paper_1101_0809_gb300.adjoint).  The kinds:

  step     pic_step on one grid, then the state read back to device arrays
  batch    an ensemble of uneven 2D runs by pic_step_graph or pic_step_persistent
  laser    a relativistic slab in a plane wave, fixed sort interval, antenna on
  monitor  pic_step with pic_diagnostics after it, as a run that logs its energy
  split    the step by its parts: pic_yee_update, pic_gather_push, pic_deposit_current
  load     pic_load_particles: absolute FP64 positions to the sorted particle store
  adjoint  value and gradients of a run's loss through torch.autograd

Units are those of the workloads: the cell is one Debye length, omega_pe = 1 and
c = v_th/(v_th/c), or c = dx = 1 for the laser.  Positions are drawn uniformly
over the box and given cell by cell, offsets and momenta as FP32 values, so that
an FP32 grid and a 64-bit one start from the same numbers.
"""
import math

import numpy as np
import torch

from paper_1101_0809_gb300 import adjoint as A
from paper_1101_0809_gb300 import pic as P

FP64, FP32 = P.PIC_FP64, P.PIC_FP32
DEV = "cuda"
F8 = torch.float64
# particle-steps, weighted by the stencil and the precision, of the largest case
LARGEST = 128 ** 3 * 64 * 12
EXACT_AT_MOST = 3.0e8   # particle-steps that the 64-bit form of a case does in reasonable time


def step(name, dims, n, ppc, **more):
    """ions: 0 a uniform background, 1836 a mobile species of that mass ratio,
    1e30 immovable ones at the electrons' positions.  tile: three extents, or 0
    for the library's own choice."""
    c = {"name": name, "kind": "step", "dims": dims, "nx": n[0], "ny": n[1], "nz": n[2] if dims == 3 else 1, "ppc": ppc,
         "fp64": False, "order2": 3, "ions": 0.0, "vth": 0.05, "courant": 0.5, "tx": 0, "ty": 0, "tz": 0, "halo": -1,
         "sort": 0, "steps": 10}
    c.update(more)
    return c


def listed():
    return [
        # the smallest run: the 2D FP64 correctness run, where launches and latency count
        step("2d_32_fp64", 2, (32, 32), 8, fp64=True, tx=8, ty=8, tz=1, steps=50),
        # the forward run of the differentiable workload: a 2D plasma in FP32
        step("2d_256_fp32", 2, (256, 256), 16, tx=16, ty=16, tz=1, steps=40),
        # the main workload: 134 M electrons and ions in 3D, three sort intervals
        step("3d_128_fp32", 3, (128, 128, 128), 32, ions=1836.0, vth=0.1, courant=0.45, tx=8, ty=4, tz=4, sort=4,
             steps=12),
        # a run that leaves tiles and sort interval to the library, on odd sizes
        step("3d_odd_default_fp32", 3, (61, 47, 53), 12, ions=1836.0, vth=0.1, courant=0.45, steps=20),
        # the plain FP64 method in 3D
        step("3d_48_fp64", 3, (48, 48, 48), 16, ions=1836.0, vth=0.1, courant=0.45, fp64=True, tx=8, ty=4, tz=4, sort=4,
             steps=4),
        # the energy experiment: few particles per cell, ions that do not move
        step("3d_64_sparse_fp32", 3, (64, 64, 64), 2, ions=1.0e30, vth=0.05, tx=8, ty=4, tz=4, steps=20),
        # the higher alternating order 2 1/2, with its own tiles and sort interval
        step("3d_64_order5_fp32", 3, (64, 64, 64), 32, ions=1836.0, vth=0.1, courant=0.45, order2=5, tx=4, ty=4, tz=4,
             sort=6, steps=6),
        # independent 2D runs of uneven size, replayed from CUDA graphs
        {"name": "batch_24_graph", "kind": "batch", "runs": 24, "nlo": 32, "nhi": 256, "plo": 4, "phi": 64, "graph": True,
         "tile": 16, "ppb": 8192, "sort": 5, "steps": 30, "pick": 3},
        # the laser slab at a fixed sort interval: strong drift and load imbalance
        {"name": "laser_slab", "kind": "laser", "nx": 256, "ny": 64, "nz": 64, "ppc": 16, "a0": 5.0, "tx": 4, "ty": 4,
         "tz": 4, "halo": 2, "sort": 10, "steps": 10},
        # a run that writes its energy integral every few steps
        {**step("monitor_96_fp32", 3, (96, 96, 96), 8, ions=1836.0, vth=0.1, courant=0.45, tx=8, ty=4, tz=4, sort=4,
                steps=4), "kind": "monitor"},
        # initial conditions into the particle store
        {"name": "load_16m", "kind": "load", "dims": 3, "nx": 80, "ny": 80, "nz": 80, "count": 16_000_000, "fp64": False,
         "order2": 3, "tx": 8, "ty": 4, "tz": 4},
        # value and gradients of the differentiable run, checkpointed
        {"name": "adjoint_256_fp32", "kind": "adjoint", "n": 256, "ppc": 16, "vth": 0.05, "fp64": False, "tile": 16,
         "steps": 40, "every": 20},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _weight(c):
    """Particle-steps of a step case in units of the l_a = 1 1/2 FP32 ones."""
    species = 1 if c["ions"] == 0 else 2
    return (c["nx"] * c["ny"] * c["nz"] * c["ppc"] * species * c["steps"] * (20.0 if c["fp64"] else 1.0)
            * (2.6 if c["order2"] == 5 else 1.0))


def _draw_step2(rng):
    t = rng.choice([(0, 0), (8, 8), (16, 16)])
    return step("", 2, (_log(rng, 28, 700), _log(rng, 28, 700)), _log(rng, 4, 48), fp64=rng.random() < 0.3,
                vth=rng.choice([0.05, 0.1]), ions=rng.choice([0.0, 0.0, 1836.0]), tx=t[0], ty=t[1],
                sort=rng.choice([0, 4, 6]), steps=rng.randint(10, 50))


def _draw_step3(rng):
    order2 = rng.choice([3, 3, 3, 5])
    t = (4, 4, 4) if order2 == 5 else rng.choice([(0, 0, 0), (8, 4, 4), (8, 4, 4)])
    return step("", 3, tuple(_log(rng, 20, 128) for _ in range(3)), _log(rng, 2, 32), order2=order2,
                fp64=rng.random() < 0.2, ions=rng.choice([0.0, 1836.0, 1836.0, 1.0e30]), vth=rng.choice([0.05, 0.1]),
                courant=0.45, tx=t[0], ty=t[1], tz=t[2], sort=rng.choice([0, 4, 6]), steps=rng.randint(4, 20))


def draw(rng):
    kind = rng.choice(["step2", "step3", "step3", "batch", "laser", "monitor", "split", "load", "adjoint"])
    while True:
        if kind in ("step2", "step3", "monitor", "split"):
            c = _draw_step2(rng) if kind == "step2" else _draw_step3(rng)
            if kind == "step2" and rng.random() < 0.3:
                kind = "split"
            if kind == "split":
                c["steps"] = min(c["steps"], 10)
            c["kind"] = kind if kind in ("monitor", "split") else "step"
            c.pop("name")
            if 2.0e5 < _weight(c) <= LARGEST / 2:
                return c
            kind = "step2" if c["dims"] == 2 else c["kind"].replace("step", "step3")
            continue
        if kind == "batch":
            lo, hi = _log(rng, 26, 64), _log(rng, 96, 256)
            graph = rng.random() < 0.5
            sort = rng.randint(3, 6)
            return {"kind": "batch", "runs": rng.randint(4, 32), "nlo": lo, "nhi": hi, "plo": 4, "phi": _log(rng, 8, 64),
                    "graph": graph, "tile": rng.choice([8, 16]), "ppb": rng.choice([2048, 4096, 8192]), "sort": sort,
                    "steps": 2 * sort * rng.randint(2, 4) if graph else rng.randint(10, 30),
                    "pick": rng.randint(1, 1 << 20)}
        if kind == "laser":
            t = rng.choice([(8, 4, 4, 1), (4, 4, 4, 2)])
            return {"kind": "laser", "nx": rng.randint(160, 320), "ny": rng.randint(20, 72), "nz": rng.randint(20, 72),
                    "ppc": rng.randint(4, 16), "a0": rng.choice([2.0, 5.0]), "tx": t[0], "ty": t[1], "tz": t[2],
                    "halo": t[3], "sort": rng.choice([4, 10]), "steps": rng.randint(8, 20)}
        if kind == "load":
            dims = rng.choice([2, 3])
            n = (_log(rng, 64, 512), _log(rng, 64, 512), 1) if dims == 2 else tuple(_log(rng, 24, 128) for _ in range(3))
            t = rng.choice([(0, 0, 0), (8, 4, 4)]) if dims == 3 else rng.choice([(0, 0, 0), (8, 8, 1)])
            return {"kind": "load", "dims": dims, "nx": n[0], "ny": n[1], "nz": n[2], "count": _log(rng, 1000, 30_000_000),
                    "fp64": rng.random() < 0.3, "order2": 3, "tx": t[0], "ty": t[1], "tz": t[2]}
        n = _log(rng, 40, 300)
        return {"kind": "adjoint", "n": n, "ppc": rng.randint(4, 16), "vth": 0.05, "fp64": n < 100 and rng.random() < 0.4,
                "tile": rng.choice([8, 16]), "steps": rng.randint(10, 40), "every": rng.choice([10, 20])}


# ---- inputs -------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 7919 + 1101)
    return g


def _by_cell(g, dims, n, count):
    """count positions, uniform over the box, given cell by cell: three
    contiguous rows of FP64."""
    nz = n[2] if dims == 3 else 1
    cell = torch.randint(n[0] * n[1] * nz, (count,), generator=g, device=DEV, dtype=torch.int32).sort().values
    x = torch.zeros((3, count), dtype=F8, device=DEV)
    for a, idx in enumerate((cell % n[0], (cell // n[0]) % n[1], cell // (n[0] * n[1]))[:dims]):
        x[a] = idx
        x[a] += torch.rand(count, generator=g, device=DEV)
    return x


def _slab_area(span):
    """Planes' worth of full density: a linear ramp over the first 50 planes."""
    return span - 25.0 if span > 50 else span * span / 100.0


def _normal(g, count, sigma):
    w = torch.randn((3, count), generator=g, device=DEV)
    return (w * sigma).to(F8)


def _params(c):
    """Grid and run parameters of the step, monitor and split cases."""
    n = (c["nx"], c["ny"], c["nz"])
    vc = 1.0 / c["vth"]
    weight = 1.0 / (4.0 * math.pi * c["ppc"])
    return {"dims": c["dims"], "n": n, "d": (1.0, 1.0, 1.0), "dt": c["courant"] / vc, "c": vc, "weight": weight,
            "rho_bg": weight * c["ppc"] if c["ions"] == 0 else 0.0, "order2": c["order2"], "antenna": None}


def _plasma(c, seed):
    """[(q, m, weight, x, w)] of a thermal plasma."""
    p, g = _params(c), _gen(seed)
    count = c["nx"] * c["ny"] * c["nz"] * c["ppc"]
    x = _by_cell(g, c["dims"], p["n"], count)
    species = [(-1.0, 1.0, p["weight"], x, _normal(g, count, 1.0))]
    if c["ions"] >= 1.0e20:
        species.append((1.0, c["ions"], p["weight"], x, torch.zeros_like(x)))
    elif c["ions"] > 0:
        species.append((1.0, c["ions"], p["weight"], _by_cell(g, c["dims"], p["n"], count),
                        _normal(g, count, 1.0 / math.sqrt(c["ions"]))))
    return p, species, None


def _laser(c, seed):
    """Electrons of a slab in a plane wave that has already crossed it: momenta
    of a cold electron in the wave, w_y = a and w_x = a^2/2, with the wave's own
    fields on the grid (B half a step earlier), and the antenna still driving."""
    g = _gen(seed)
    n, dt, omega = (c["nx"], c["ny"], c["nz"]), 0.45, 2.0 * math.pi / 20.0
    weight = 0.01 * omega * omega / (4.0 * math.pi) / c["ppc"]
    lo, hi, plane = n[0] // 4, (3 * n[0]) // 4, 8
    count = int(_slab_area(hi - lo) * n[1] * n[2] * c["ppc"])
    u = _slab_area(hi - lo) * torch.rand(count, generator=g, device=DEV, dtype=F8)
    along = torch.where(u < 25.0, 10.0 * torch.sqrt(u), u + 25.0).clamp(max=hi - lo - 1e-6) + lo
    x = torch.stack([along, n[1] * torch.rand(count, generator=g, device=DEV, dtype=F8),
                     n[2] * torch.rand(count, generator=g, device=DEV, dtype=F8)])
    cell = torch.floor(x)
    x = cell + (x - cell).float().clamp(max=1.0 - 2.0 ** -24).to(F8)
    x = x[:, torch.argsort(cell[0] + n[0] * (cell[1] + n[1] * cell[2]), stable=True)].contiguous()
    clock = int(n[0] / dt)   # the front has gone past the far end of the slab
    t0 = clock * dt
    amplitude = c["a0"] * omega
    a = c["a0"] * torch.cos(omega * (t0 - 0.5 * dt - (x[0] - plane)))
    w = torch.zeros_like(x)
    w[0], w[1] = (0.5 * a * a).float(), a.float()
    w[2] = 0.01 * torch.randn(x.shape[1], generator=g, device=DEV)
    xs = torch.arange(n[0], dtype=F8, device=DEV)
    inside = (xs >= plane).to(F8)

    def wave(at, t):
        return (amplitude * torch.sin(omega * (t - (at - plane))) * inside).float().expand(n[2], n[1], n[0]).contiguous()

    zero = torch.zeros((n[2], n[1], n[0]), device=DEV)
    fields = ([zero, wave(xs + 0.5, t0), zero], [zero, zero, wave(xs, t0 - 0.5 * dt)])
    p = {"dims": 3, "n": n, "d": (1.0, 1.0, 1.0), "dt": dt, "c": 1.0, "weight": weight, "rho_bg": 0.0, "order2": 3,
         "antenna": {"plane": plane, "amplitude": amplitude, "omega": omega, "ramp": 40.0, "start": clock}}
    return p, [(-1.0, 1.0, weight, x, w)], fields


def _desc(c, p, stream=None):
    return P.make_desc(p["dims"], p["n"], p["d"], p["dt"], p["c"], FP64 if c.get("fp64") else FP32,
                       tile=(c["tx"], c["ty"], c["tz"]), halo=c.get("halo", -1), sort_interval=c.get("sort", 0),
                       rho_bg=p["rho_bg"], order2=p["order2"], stream=stream)


class _Read:
    """Device arrays that a run's state is read back into."""

    def __init__(self, c, p, counts):
        self.n, self.dims, self.fp64 = p["n"], p["dims"], bool(c.get("fp64"))
        dt = F8 if self.fp64 else torch.float32
        shape = (p["n"][2] if p["dims"] == 3 else 1, p["n"][1], p["n"][0])
        # a vector's components are parts of one array, as a program that compares vectors holds them
        self.fields = [torch.empty((3, *shape), dtype=dt, device=DEV) for _ in range(3)]
        self.species = [(torch.empty(m, dtype=torch.int32, device=DEV), torch.empty(m, dtype=torch.int32, device=DEV),
                         torch.empty((p["dims"], m), dtype=dt, device=DEV), torch.empty((3, m), dtype=dt, device=DEV))
                        for m in counts]

    def order_of_ids(self, k, cell, ident, off, w, x0):
        """Positions and momenta by particle id, each position as the image that
        lies nearest to where its particle was loaded."""
        idx = ident.long()
        nx, ny = self.n[0], self.n[1]
        x, wid = torch.empty_like(off), torch.empty_like(w)
        at = cell
        for a in range(self.dims):
            along = at if a == self.dims - 1 else at % self.n[a]
            if a < self.dims - 1:
                at = torch.div(at, (nx, ny)[a], rounding_mode="floor")
            x[a][idx] = off[a] + along
            x[a].sub_(torch.round((x[a] - x0[k][a]) / self.n[a]), alpha=self.n[a])
        for a in range(3):
            wid[a][idx] = w[a]
        return {"x": x, "w": wid}

    def all(self, grid, x0):
        E, B, J = self.fields
        P.pic_get_fields(grid.h, list(E), list(B), list(J))
        species = []
        for k, (cell, ident, off, w) in enumerate(self.species):
            P.pic_get_particles(grid.h, k, cell, list(off) if self.dims == 3 else [off[0], off[1], None], list(w), ident)
            # an FP64 state comes as the library stores it, an FP32 one by id
            species.append({"cell": cell, "id": ident, "offset": off, "w": w} if self.fp64
                           else self.order_of_ids(k, cell, ident, off, w, x0))
        return {"E": E, "B": B, "J": J, "species": species}


class _State:
    pass


def prepare(case, seed):
    c = dict(case)
    kind = c["kind"]
    s = _State()
    s.c = c
    if kind == "batch":
        return _prepare_batch(s, c, seed)
    if kind == "adjoint":
        return _prepare_adjoint(s, c, seed)
    if kind == "load":
        n = (c["nx"], c["ny"], c["nz"])
        g = _gen(seed)
        s.p = {"dims": c["dims"], "n": n, "d": (1.0,) * 3, "dt": 0.02, "c": 20.0, "rho_bg": 0.0, "order2": 3}
        x = torch.rand((3, c["count"]), generator=g, device=DEV, dtype=F8)
        s.x = [(x[a] * n[a]).contiguous() for a in range(3)]
        s.w = list(torch.randn((3, c["count"]), generator=g, device=DEV, dtype=F8))
        s.grid = P.Grid(_desc(c, s.p))
        s.read = _Read(c, s.p, [c["count"]])
        torch.cuda.synchronize()
        return s
    s.p, species, fields = _laser(c, seed) if kind == "laser" else _plasma(c, seed)
    s.grid = P.Grid(_desc(c, s.p))
    if fields:
        P.pic_set_fields(s.grid.h, fields[0], fields[1])
    s.x0 = []
    for k, (q, m, weight, x, w) in enumerate(species):
        P.pic_load_particles(s.grid.h, k, q, m, weight, list(x), list(w))
        s.x0.append(x.float() if not c.get("fp64") else None)
    if s.p["antenna"]:
        a = s.p["antenna"]
        P.pic_set_antenna(s.grid.h, 0, P.PIC_POL_Y, a["plane"], a["amplitude"], a["omega"], a["ramp"], a["start"])
    s.read = _Read(c, s.p, [sp[3].shape[1] for sp in species])
    torch.cuda.synchronize()
    return s


def _runs(c, seed):
    """Sizes from the case, inputs from the seed: the batch's runs."""
    r = np.random.Generator(np.random.PCG64(c["pick"]))
    g = _gen(seed)
    out = []
    for _ in range(c["runs"]):
        n, ppc, vth = int(r.integers(c["nlo"], c["nhi"] + 1)), int(r.integers(c["plo"], c["phi"] + 1)), float(r.uniform(0.01, 0.3))
        weight = vth * vth / (4.0 * math.pi * ppc)
        p = {"dims": 2, "n": (n, n, 1), "d": (1.0,) * 3, "dt": 0.5, "c": 1.0, "weight": weight, "rho_bg": weight * ppc,
             "order2": 3, "antenna": None}
        out.append((p, [(-1.0, 1.0, weight, _by_cell(g, 2, (n, n), n * n * ppc), _normal(g, n * n * ppc, vth))]))
    return out


def _prepare_batch(s, c, seed):
    runs = _runs(c, seed)
    s.stream = torch.cuda.Stream()
    descs = [P.make_desc(2, p["n"], p["d"], p["dt"], p["c"], FP32, tile=(c["tile"], c["tile"], 1), halo=1,
                         sort_interval=c["sort"], particles_per_block=c["ppb"], rho_bg=p["rho_bg"],
                         stream=s.stream.cuda_stream) for p, _ in runs]
    s.grid = P.Batch(descs)
    torch.cuda.synchronize()
    P.pic_load_particles_runs(s.grid.h, list(range(len(runs))), 0, [sp[0][:3] for _, sp in runs],
                              [list(sp[0][3]) for _, sp in runs], [list(sp[0][4]) for _, sp in runs])
    # every run's arrays are parts of one: the fields run after run, then the particles
    s.shapes = [(1, p["n"][1], p["n"][0]) for p, _ in runs]
    cells = [a[1] * a[2] for a in s.shapes]
    counts = [sp[0][3].shape[1] for _, sp in runs]
    s.fields = [torch.empty((3, sum(cells)), device=DEV) for _ in range(3)]
    s.parts = [[[t.view(a) for t, a in zip(f.split(cells), s.shapes)] for f in fs] for fs in s.fields]
    s.off = torch.empty((2, sum(counts)), device=DEV)
    s.w = torch.empty((3, sum(counts)), device=DEV)
    s.cell, s.id = (torch.empty(sum(counts), dtype=torch.int32, device=DEV) for _ in range(2))
    s.bits = [t.split(counts) for t in (s.cell, s.id, *s.off, *s.w)]
    s.first = torch.tensor(np.repeat(np.cumsum([0] + counts[:-1]), counts), device=DEV)
    s.width = torch.tensor(np.repeat([p["n"][0] for p, _ in runs], counts), dtype=torch.int32, device=DEV)
    s.x0 = [torch.cat([sp[0][3][a] for _, sp in runs]).float() for a in range(2)]
    torch.cuda.synchronize()
    return s


def _prepare_adjoint(s, c, seed):
    """The differentiable run: a sinusoidal density perturbation of 5 percent,
    the field energy of a window as its loss."""
    g = _gen(seed)
    n, vc = c["n"], 1.0 / c["vth"]
    weight = 1.0 / (4.0 * math.pi * c["ppc"])
    x = _by_cell(g, 2, (n, n), n * n * c["ppc"])
    k = 4.0 * math.pi / n
    x[0] = torch.remainder(x[0] - (0.05 / k) * torch.sin(k * x[0]), float(n))
    x[0][x[0] >= n] = 0.0
    s.p = {"dims": 2, "n": (n, n, 1), "d": (1.0,) * 3, "dt": 0.5 / vc, "c": vc, "weight": weight, "rho_bg": weight * c["ppc"],
           "order2": 3, "antenna": None}
    s.x, s.w = x, _normal(g, x.shape[1], 1.0)
    at = n // 4
    s.window = ((at, at + min(32, n // 2)), (at, at + min(32, n // 2)))
    desc = P.make_desc(2, s.p["n"], s.p["d"], s.p["dt"], vc, FP64 if c["fp64"] else FP32, tile=(c["tile"], c["tile"], 1),
                       rho_bg=s.p["rho_bg"])
    s.run = A.DifferentiableRun(desc, -1.0, 1.0, weight, c["steps"], s.window, c["every"])
    torch.cuda.synchronize()
    return s


# ---- one pass --------------------------------------------------------------------------

def run(s):
    c, kind = s.c, s.c["kind"]
    if kind == "adjoint":
        x, w = s.x.clone().requires_grad_(), s.w.clone().requires_grad_()
        loss = A.WindowEnergyLoss.apply(x, w, s.run)
        loss.backward()
        if c["fp64"]:
            return {"loss": loss.detach(), "gx": x.grad, "gw": w.grad}
        return {"loss": loss.detach().float(), "gx": x.grad.float(), "gw": w.grad.float()}
    if kind == "batch":
        return _run_batch(s, c)
    g = s.grid.h
    if kind == "load":
        P.pic_load_particles(g, 0, -1.0, 1.0, 1.0, s.x, s.w)
        cell, ident, off, w = s.read.species[0]
        P.pic_get_particles(g, 0, cell, list(off) if c["dims"] == 3 else [off[0], off[1], None], list(w), ident)
        return {"cell": cell, "id": ident, "offset": off, "w": w}
    if kind == "split":
        for k in range(c["steps"]):
            if k % 5 == 0:
                P.pic_sort(g)
            P.pic_yee_update(g, P.PIC_B_HALF)
            P.pic_gather_push(g)
            P.pic_deposit_current(g)
            P.pic_yee_update(g, P.PIC_B_HALF)
            P.pic_yee_update(g, P.PIC_E_FULL)
    else:
        P.pic_step(g, c["steps"])
    if kind == "monitor":
        d = P.pic_diagnostics(g)
        E, B, J = s.read.fields
        P.pic_get_fields(g, list(E), list(B), list(J))
        log = np.array([d["kinetic"], d["field_E"], d["field_B"], d["half_step_corr"], d["total"], *d["momentum"],
                        d["total_charge"]], dtype=np.float64 if c["fp64"] else np.float32)
        return {"log": log, "E": E, "B": B, "J": J}
    return s.read.all(s.grid, s.x0)


def _run_batch(s, c):
    h = s.grid.h
    with torch.cuda.stream(s.stream):
        (P.pic_step_graph if c["graph"] else P.pic_step_persistent)(h, c["steps"])
        for r in range(c["runs"]):
            P.pic_get_fields_run(h, r, *[[f[r] for f in fs] for fs in s.parts])
            cell, ident, o0, o1, w0, w1, w2 = (b[r] for b in s.bits)
            P.pic_get_particles_run(h, r, 0, cell, [o0, o1, None], [w0, w1, w2], ident)
        idx = s.first + s.id
        x, w = torch.empty_like(s.off), torch.empty_like(s.w)
        for a, along in enumerate((s.cell % s.width, torch.div(s.cell, s.width, rounding_mode="floor"))):
            x[a][idx] = s.off[a] + along
            x[a].sub_(s.width * torch.round((x[a] - s.x0[a]) / s.width))
        for a in range(3):
            w[a][idx] = s.w[a]
    torch.cuda.current_stream().wait_stream(s.stream)
    return {"E": s.fields[0], "B": s.fields[1], "J": s.fields[2], "x": x, "w": w}


# ---- what a pass cannot do without ------------------------------------------------------

def work(case):
    """State in and out once per step (the sort and the read-back left out), and
    the operations of gather, push and deposit per particle and step."""
    c = case
    kind = c["kind"]
    es = 8 if c.get("fp64") else 4
    if kind == "load":
        d = c["dims"]
        return {"bytes": c["count"] * (8 * (d + 3) + 8 + es * (d + 3)), "flops": c["count"] * 4 * d}
    if kind == "batch":
        r = np.random.Generator(np.random.PCG64(c["pick"]))
        b = f = 0
        for _ in range(c["runs"]):
            n, ppc = int(r.integers(c["nlo"], c["nhi"] + 1)), int(r.integers(c["plo"], c["phi"] + 1))
            r.uniform(0.01, 0.3)
            b += n * n * (ppc * 48 + 120)
            f += n * n * (ppc * 330 + 40)
        return {"bytes": b * c["steps"], "flops": f * c["steps"]}
    if kind == "adjoint":
        m, cells = c["n"] ** 2 * c["ppc"], c["n"] ** 2
        return {"bytes": c["steps"] * es * (m * (12 + 12 + 16) + cells * 60), "flops": c["steps"] * m * 1400}
    if kind == "laser":
        m = int(_slab_area((3 * c["nx"]) // 4 - c["nx"] // 4) * c["ny"] * c["nz"] * c["ppc"])
        cells, d, order2 = c["nx"] * c["ny"] * c["nz"], 3, 3
    else:
        cells = c["nx"] * c["ny"] * c["nz"]
        species = 1 if c["ions"] == 0 else 2
        m, d, order2 = cells * c["ppc"] * species, c["dims"], c["order2"]
    per = (330 if d == 2 else 700) * (2.6 if order2 == 5 else 1.0)
    bytes_ = c["steps"] * (m * 2 * (4 + es * (d + 3)) + cells * 30 * es)
    if kind == "monitor":
        bytes_ += m * (4 + es * (d + 3)) + cells * 6 * es
    return {"bytes": bytes_, "flops": c["steps"] * (m * per + cells * 60)}


# ---- the same in 64 bits, by plain torch -------------------------------------------------

def _weights(x, order2):
    """Base index, the point weights f and the cell weights S of the alternating
    order, each with the offset of its first entry from the base."""
    if order2 == 5:
        ib = torch.floor(x + 0.5)
        d = x + 0.5 - ib
        e = 1 - d
        f = [e * e / 2, 0.75 - (0.5 - d) ** 2, d * d / 2]
        S = [e ** 3 / 6, (4 - 6 * d ** 2 + 3 * d ** 3) / 6, (1 + 3 * d + 3 * d ** 2 - 3 * d ** 3) / 6, d ** 3 / 6]
        return ib, f, -1, S, -2
    ib = torch.floor(x)
    d = x - ib
    return ib, [1 - d, d], 0, [(1 - d) ** 2 / 2, 0.75 - (0.5 - d) ** 2, d * d / 2], -1


def _flat(n, dims, at):
    i = torch.remainder(at[0], n[0]) + n[0] * torch.remainder(at[1], n[1])
    return i + n[0] * n[1] * torch.remainder(at[2], n[2]) if dims == 3 else i


def _gather(p, F, x, magnetic):
    """F (three flat arrays) at the particles: alpha (E) or beta (B) weights."""
    dims, n = p["dims"], p["n"]
    sets = [_weights(x[a], p["order2"]) for a in range(dims)]
    ib = [s[0].long() for s in sets]
    out = []
    for comp in range(3):
        per = []
        for a in range(dims):
            _, f, f0, S, S0 = sets[a]
            point = (a == comp) != magnetic
            per.append([(f0 + q, v) for q, v in enumerate(f)] if point else [(S0 + q, v) for q, v in enumerate(S)])
        total = torch.zeros_like(x[0])
        for oy, vy in per[1]:
            for oz, vz in (per[2] if dims == 3 else [(0, None)]):
                vyz = vy * vz if dims == 3 else vy
                for ox, vx in per[0]:
                    at = [ib[0] + ox, ib[1] + oy] + ([ib[2] + oz] if dims == 3 else [])
                    total = total + vx * vyz * F[comp][_flat(n, dims, at)]
        out.append(total)
    return out


def _deposit(p, J, qp, x0, x1, uz):
    """Adds the virtual-path current of x0 -> x1 to J (three flat arrays)."""
    dims, n, V = p["dims"], p["n"], 1.0
    win, lo, ib = [], [], []
    for a in range(dims):
        b0, _, _, S0, o0 = _weights(x0[a], p["order2"])
        b1, _, _, S1, _ = _weights(x1[a], p["order2"])
        sh = (b1 - b0).long()
        k = len(S0)
        zero = torch.zeros_like(S0[0])
        old = [zero] + S0 + [zero]
        new = [torch.where(sh < 0, S1[q] if q < k else zero, torch.where(sh == 0, S1[q - 1] if 1 <= q <= k else zero,
                                                                         S1[q - 2] if q >= 2 else zero)) for q in range(k + 2)]
        Pp, Pm = [u + v for u, v in zip(new, old)], [u - v for u, v in zip(new, old)]
        D, run_ = [], zero
        for q in range(k + 1):
            run_ = run_ + Pm[q]
            D.append(run_)
        win.append((Pp, Pm, D))
        lo.append(o0 - 1)
        ib.append(b0.long())

    def add(comp, at, v):
        J[comp] = J[comp].index_add(0, _flat(n, dims, at), v) if v.requires_grad else J[comp].index_add_(0, _flat(n, dims, at), v)

    m = len(win[0][0])
    if dims == 2:
        (Px, Mx, Dx), (Py, My, Dy) = win
        for w in range(m):
            for q in range(m - 1):
                add(0, [ib[0] + lo[0] + 1 + q, ib[1] + lo[1] + w], (-0.5 / p["dt"] * qp / V) * Dx[q] * Py[w])
                add(1, [ib[0] + lo[0] + w, ib[1] + lo[1] + 1 + q], (-0.5 / p["dt"] * qp / V) * Dy[q] * Px[w])
            for v in range(m):
                add(2, [ib[0] + lo[0] + w, ib[1] + lo[1] + v],
                    (0.25 * qp / V) * uz * (Px[w] * Py[v] + Mx[w] * My[v] / 3))
        return
    for comp in range(3):
        b, c = [a for a in range(3) if a != comp]
        for wb in range(m):
            for wc in range(m):
                T = win[b][0][wb] * win[c][0][wc] + win[b][1][wb] * win[c][1][wc] / 3
                for q in range(m - 1):
                    at = [None] * 3
                    at[comp] = ib[comp] + lo[comp] + 1 + q
                    at[b] = ib[b] + lo[b] + wb
                    at[c] = ib[c] + lo[c] + wc
                    add(comp, at, (-0.25 / p["dt"] * qp / V) * win[comp][2][q] * T)


def _dm(f, axis):
    return f - torch.roll(f, 1, 2 - axis)


def _dp(f, axis):
    return torch.roll(f, -1, 2 - axis) - f


def _incident(a, p, at, t):
    tau = t - (at - a["plane"]) / p["c"]
    if tau <= 0.0:
        return 0.0
    g = math.sin(0.5 * math.pi * tau / a["ramp"]) ** 2 if tau < a["ramp"] else 1.0
    return a["amplitude"] * g * math.sin(a["omega"] * tau)


def _b_half(p, E, B, clock):
    h = 0.5 * p["c"] * p["dt"]
    bx, by, bz = B[0] - h * _dm(E[2], 1), B[1] + h * _dm(E[2], 0), B[2] - h * _dm(E[1], 0) + h * _dm(E[0], 1)
    if p["dims"] == 3:
        bx, by = bx + h * _dm(E[1], 2), by - h * _dm(E[0], 2)
    if p["antenna"]:
        a = p["antenna"]
        bz = bz.clone()
        bz[:, :, a["plane"]] += h * _incident(a, p, a["plane"] - 0.5, clock * p["dt"])
    return [bx, by, bz]


def _e_full(p, E, B, J, clock):
    h, f = p["c"] * p["dt"], 4.0 * math.pi * p["dt"]
    ex, ey = E[0] - f * J[0] + h * _dp(B[2], 1), E[1] - f * J[1] - h * _dp(B[2], 0)
    ez = E[2] - f * J[2] + h * _dp(B[1], 0) - h * _dp(B[0], 1)
    if p["dims"] == 3:
        ex, ey = ex - h * _dp(B[1], 2), ey + h * _dp(B[0], 2)
    if p["antenna"]:
        a = p["antenna"]
        ey = ey.clone()
        ey[:, :, a["plane"] - 1] += h * _incident(a, p, a["plane"], (clock + 0.5) * p["dt"])
    return [ex, ey, ez]


def _exact_step(p, E, B, species, clock=0, chunk=1 << 22):
    """One step; species: [q, m, weight, x (list), w (list)], advanced in place
    of the lists.  Positions stay unwrapped.  Returns E, B, J."""
    shape = E[0].shape
    B = _b_half(p, E, B, clock)
    Ef, Bf = [f.reshape(-1) for f in E], [f.reshape(-1) for f in B]
    J = [torch.zeros(shape.numel(), dtype=F8, device=DEV) for _ in range(3)]
    for sp in species:
        q, m, weight, xs, ws = sp
        many = [torch.split(v, chunk) for v in (*xs, *ws)]
        done = []
        for part in zip(*many):
            x, w = list(part[:p["dims"]]), list(part[p["dims"]:])
            Ep, Bp = _gather(p, Ef, x, False), _gather(p, Bf, x, True)
            h = 0.5 * q / m * p["dt"]
            e = [h * v for v in Ep]
            t = [u + v for u, v in zip(w, e)]
            s = h / torch.sqrt(t[0] ** 2 + t[1] ** 2 + t[2] ** 2 + p["c"] ** 2)
            b = [s * v for v in Bp]
            cross = lambda u, v: [u[1] * v[2] - u[2] * v[1], u[2] * v[0] - u[0] * v[2], u[0] * v[1] - u[1] * v[0]]  # noqa: E731
            nn = [u + v for u, v in zip(t, cross(t, b))]
            f = 2.0 / (1.0 + b[0] ** 2 + b[1] ** 2 + b[2] ** 2)
            w1 = [u + v + f * r for u, v, r in zip(t, e, cross(nn, b))]
            ig = p["c"] / torch.sqrt(w1[0] ** 2 + w1[1] ** 2 + w1[2] ** 2 + p["c"] ** 2)
            x1 = [x[a] + w1[a] * ig * p["dt"] / p["d"][a] for a in range(p["dims"])]
            _deposit(p, J, q * weight, x, x1, w1[2] * ig)
            done.append(x1 + w1)
        rows = [torch.cat(v) if len(v) > 1 else v[0] for v in zip(*done)]
        sp[3], sp[4] = rows[:p["dims"]], rows[p["dims"]:]
    J = [f.reshape(shape) for f in J]
    B = _b_half(p, E, B, clock)
    return _e_full(p, E, B, J, clock), B, J


def _exact_run(p, species, fields, steps):
    shape = (p["n"][2] if p["dims"] == 3 else 1, p["n"][1], p["n"][0])
    E, B = ([f.to(F8) for f in fs] if fs is not None else [torch.zeros(shape, dtype=F8, device=DEV) for _ in range(3)]
            for fs in (fields or (None, None)))
    sp = [[q, m, wt, list(x)[:p["dims"]], list(w)] for q, m, wt, x, w in species]
    J = None
    start = p["antenna"]["start"] if p["antenna"] else 0
    for k in range(steps):
        E, B, J = _exact_step(p, E, B, sp, start + k)
    return E, B, J, sp


def _exact_log(p, E, B, sp):
    """The energy integral and the sums beside it at the state's time level."""
    c, V = p["c"], 1.0
    Bn = _b_half({**p, "antenna": None}, E, B, 0)
    kin = half = charge = 0.0
    mom = [0.0, 0.0, 0.0]
    Ef = [f.reshape(-1) for f in E]
    for q, m, weight, x, w in sp:
        for part in zip(*[torch.split(v, 1 << 22) for v in (*x, *w)]):
            xp, wp = list(part[:p["dims"]]), list(part[p["dims"]:])
            w2 = wp[0] ** 2 + wp[1] ** 2 + wp[2] ** 2
            g = torch.sqrt(w2 + c * c)
            kin += float((m * weight * c * w2 / (g + c)).sum())
            Ep = _gather(p, Ef, xp, False)
            half += float((0.5 * q * weight * p["dt"] * c * (wp[0] * Ep[0] + wp[1] * Ep[1] + wp[2] * Ep[2]) / g).sum())
            for a in range(3):
                mom[a] += float((m * weight * wp[a]).sum())
            charge += q * weight * xp[0].numel()
    fe, fb = (V / (8.0 * math.pi) * sum(float((f ** 2).sum()) for f in F) for F in (E, Bn))
    charge += p["rho_bg"] * V * E[0].numel()
    return np.array([kin, fe, fb, half, kin + fe + fb + half, *mom, charge])


def exact(case, seed):
    c, kind = dict(case), case["kind"]
    if kind == "load":
        return None   # copied and rounded once, in whole numbers and bits
    with torch.no_grad():
        if kind == "batch":
            runs = _runs(c, seed)
            if sum(sp[0][3].shape[1] for _, sp in runs) * c["steps"] > 3 * EXACT_AT_MOST:
                return None
            got = [_exact_run(p, sp, None, c["steps"]) for p, sp in runs]
            out = {k: torch.stack([torch.cat([r[f][a].reshape(-1) for r in got]) for a in range(3)])
                   for f, k in enumerate("EBJ")}
            out["x"] = torch.stack([torch.cat([_near(r[3][0][3][a], sp[0][3][a], p["n"][a])
                                               for r, (p, sp) in zip(got, runs)]) for a in range(2)])
            out["w"] = torch.stack([torch.cat([r[3][0][4][a] for r in got]) for a in range(3)])
            return out
        if kind != "adjoint":
            p, species, fields = _laser(c, seed) if kind == "laser" else _plasma(c, seed)
            count = sum(sp[3].shape[1] for sp in species)
            if count * c["steps"] * (2.6 if p["order2"] == 5 else 1.0) > EXACT_AT_MOST * (3 if p["dims"] == 2 else 1):
                return None
            E, B, J, sp = _exact_run(p, species, fields, c["steps"])
            if kind == "monitor":
                return {"log": _exact_log(p, E, B, sp), "E": torch.stack(E), "B": torch.stack(B), "J": torch.stack(J)}
            rest = [None if c.get("fp64") else
                    {"x": torch.stack([_near(v, u, p["n"][a]) for a, (v, u) in enumerate(zip(s[3], o[3]))]),
                     "w": torch.stack(s[4])} for s, o in zip(sp, species)]
            return {"E": torch.stack(E), "B": torch.stack(B), "J": torch.stack(J), "species": rest}
    s = _State()
    s = _prepare_adjoint(s, c, seed)
    if s.x.shape[1] * c["steps"] > EXACT_AT_MOST / 4:
        return None
    return _exact_gradient(s, c)


def _near(x, x0, n):
    return x - n * torch.round((x - x0) / n)


def _exact_gradient(s, c):
    """Reverse mode through the 64-bit step, one step's graph at a time."""
    p, n = s.p, s.p["n"][0]
    shape = (1, n, n)
    E = [torch.zeros(shape, dtype=F8, device=DEV) for _ in range(3)]
    B = [f.clone() for f in E]
    x, w = [s.x[a].clone() for a in range(2)], [s.w[a].clone() for a in range(3)]
    levels = []
    with torch.no_grad():
        for _ in range(c["steps"]):
            levels.append([*E, *B, *x, *w])
            sp = [[-1.0, 1.0, p["weight"], x, w]]
            E, B, _ = _exact_step(p, E, B, sp, chunk=1 << 30)
            x, w = sp[0][3], sp[0][4]
    (x0, x1), (y0, y1) = s.window
    leaf = [f.detach().requires_grad_() for f in (*E, *B)]
    Bn = _b_half(p, leaf[:3], leaf[3:], 0)
    loss = sum((f[:, y0:y1, x0:x1] ** 2).sum() for f in (*leaf[:3], *Bn)) / (8.0 * math.pi)
    g = list(torch.autograd.grad(loss, leaf)) + [torch.zeros_like(v) for v in (*x, *w)]
    for lv in reversed(levels):
        leaf = [v.detach().requires_grad_() for v in lv]
        sp = [[-1.0, 1.0, p["weight"], leaf[6:8], leaf[8:11]]]
        E1, B1, _ = _exact_step(p, leaf[:3], leaf[3:6], sp, chunk=1 << 30)
        g = list(torch.autograd.grad([*E1, *B1, *sp[0][3], *sp[0][4]], leaf, g, allow_unused=True))
        g = [torch.zeros_like(v) if u is None else u for u, v in zip(g, leaf)]
    return {"loss": loss.detach(), "gx": torch.stack([g[6], g[7], torch.zeros_like(g[6])]), "gw": torch.stack(g[8:11])}
