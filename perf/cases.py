"""Work that users of this library have it do, for timing it and for comparing its results.

A pass is a whole request as a program makes it: the initial primitive state goes in from
page-locked host memory, a number of SSP Runge-Kutta steps run (with the host in the loop
where a program has it there), and the whole conserved state comes back to page-locked host
memory. Every pass starts from the same initial state. The sizes are those of the library's
benchmark and tests and others of the same range: grids from one block to 4096 blocks of
16^3 cells, uneven box shapes, every physics module, both stencil precisions, uniform and
refined meshes, single solves and batches.
"""
import ctypes as C
import math

import numpy as np
import torch

from paper_2607_19277_gb300 import agile
from paper_2607_19277_gb300 import workloads

NV = {"hd": 5, "mhd": 9, "srhd": 5, "ffhd": 6, "ffhd_htc": 7}
NT = {"hd": 5, "mhd": 9, "srhd": 7, "ffhd": 6, "ffhd_htc": 7}
# arithmetic of one cell in one stage (primitive recovery once, slopes once per direction,
# three faces, update), counted from the formulas
FLOPS = {"hd": 420, "mhd": 1000, "srhd": 700, "ffhd": 380, "ffhd_htc": 460}
GAMMA = {"hd": 5.0 / 3.0, "mhd": 5.0 / 3.0, "srhd": 4.0 / 3.0, "ffhd": 5.0 / 3.0, "ffhd_htc": 5.0 / 3.0}
KAPPA0 = 1e-3
TP = 2.0 * math.pi
WALLS = {"periodic": ("periodic",) * 6,
         "tube": ("outflow", "outflow", "periodic", "periodic", "periodic", "periodic"),
         "open": ("outflow",) * 6,
         "mixed": ("outflow", "reflect", "periodic", "periodic", "reflect", "reflect")}


def _case(name=None, **kw):
    c = dict(kind="mesh", physics="hd", start="waves", limiter="vanleer", flux="tvdlf", rk=3, bytes=4,
             bx=4, by=4, bz=4, walls="periodic", steps=10, host_dt=False, sums_every=0, losses=False,
             eos="ideal", levels=1, sizes="")
    assert set(kw) <= set(c)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # a small shock tube whose program sets the time step itself (the set-up of the parity
        # tests): eight blocks, launches and round trips count
        _case("tube_32_fp64_host_dt", start="tube", walls="tube", limiter="minmod", flux="hll", rk=2, bytes=8,
              bx=2, by=2, bz=2, steps=8, host_dt=True),
        # the Sod tube at 64^3, 20 steps: the smallest of the library's benchmark set-ups
        _case("tube_64_fp64", start="tube", walls="tube", limiter="minmod", flux="hll", rk=2, bytes=8, steps=20),
        # the scheme of the paper's throughput tables (hydro, TVDLF, van Leer, SSPRK3) in the
        # paper's precision, on a box of uneven block counts
        _case("shear_96x80x112_fp64", start="shear", bytes=8, bx=6, by=5, bz=7, steps=4),
        # the same scheme in the FP32 stencil at the tables' 256^3
        _case("shear_256_fp32", start="shear", bx=16, by=16, bz=16, steps=20),
        # the headline benchmark: MHD 256^3, conserved sums logged as it runs
        _case("vortex_256_mhd_fp32", physics="mhd", start="vortex", flux="hll", bx=16, by=16, bz=16, steps=20,
              sums_every=5),
        # the same in FP64 at 128^3
        _case("vortex_128_mhd_fp64", physics="mhd", start="vortex", flux="hll", bytes=8, bx=8, by=8, bz=8, steps=2),
        # a small MHD solve between walls, as a stream of small requests has it
        _case("waves_48x80x32_mhd_fp32", physics="mhd", flux="hll", limiter="minmod", rk=2, walls="mixed", bx=3, by=5,
              bz=2, steps=25),
        # a blast on an octree of 16^3 blocks: mesh set-up, refinement by the estimator, steps
        # with coarse-fine ghosts and flux correction
        _case("blast_amr4_hd_fp32", kind="amr", start="blast", walls="open", limiter="minmod", flux="hll", rk=2,
              levels=4, steps=16),
        # the same for MHD on a periodic box of uneven block counts
        _case("blast_amr3_mhd_fp32", kind="amr", physics="mhd", start="blast", flux="hll", bx=3, by=4, bz=2,
              levels=3, steps=10),
        # relativistic shells: a running batch of solves from 32^3 to 128^3; one of them leaves
        # and another joins half way
        _case("shells_batch12_srhd_fp32", kind="batch", physics="srhd", start="shell", rk=2, steps=10,
              sizes="2,8,3,4,6,2,5,4,3,7,2,4"),
        # one relativistic solve in FP64
        _case("shell_48x64x80_srhd_fp64", physics="srhd", start="shell", rk=2, bytes=8, bx=3, by=4, bz=5, steps=5),
        # field-aligned hydrodynamics with thermal conduction and radiative losses
        _case("loop_112x96x160_ffhd_fp32", physics="ffhd_htc", start="loop", bx=7, by=6, bz=10, steps=12,
              losses=True),
    ]


def _box(rng, lo, hi):
    """Block counts whose product is log-uniform between lo and hi, no side over 16."""
    n = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    bx = max(1, min(16, round(n ** (1 / 3) * math.exp(rng.uniform(-0.5, 0.5)))))
    by = max(1, min(16, round(math.sqrt(n / bx) * math.exp(rng.uniform(-0.3, 0.3)))))
    return bx, by, max(1, min(16, round(n / bx / by)))


def draw(rng):
    kind = rng.choice(["mesh"] * 5 + ["amr", "batch"])
    limiter = rng.choice(["minmod", "vanleer"])
    rk = rng.choice([2, 3])
    if kind == "batch":
        physics = rng.choice(["hd", "mhd", "srhd", "srhd"])
        sizes = [round(math.exp(rng.uniform(math.log(2), math.log(8)))) for _ in range(rng.randint(3, 12))]
        return _case(kind=kind, physics=physics, limiter=limiter, rk=rk, steps=rng.randint(6, 10),
                     start="shell" if physics == "srhd" else "waves",
                     flux="tvdlf" if physics == "srhd" else rng.choice(["tvdlf", "hll"]),
                     bytes=rng.choice([4, 4, 4, 8]) if sum(s ** 3 for s in sizes) < 600 else 4,
                     eos="synge" if physics == "srhd" and rng.random() < 0.3 else "ideal",
                     sizes=",".join(str(s) for s in sizes))
    if kind == "amr":
        physics = rng.choice(["hd", "hd", "mhd"])
        bx, by, bz = _box(rng, 8, 64)
        return _case(kind=kind, physics=physics, start="blast", limiter=limiter, rk=rk, steps=rng.randint(4, 12),
                     flux=rng.choice(["tvdlf", "hll"]), bytes=rng.choice([4, 4, 8]), bx=bx, by=by, bz=bz,
                     levels=3, walls=rng.choice(["periodic", "open"]))
    physics = rng.choice(["hd", "hd", "mhd", "mhd", "srhd", "ffhd", "ffhd_htc"])
    nbytes = rng.choice([4, 4, 8])
    bx, by, bz = _box(rng, 1, 2000 if nbytes == 4 else 250)
    start = {"hd": rng.choice(["shear", "waves", "tube"]), "mhd": rng.choice(["vortex", "waves"]), "srhd": "shell",
             "ffhd": "loop", "ffhd_htc": "loop"}[physics]
    flux = {"hd": rng.choice(["tvdlf", "hll", "hllc"]), "mhd": rng.choice(["tvdlf", "hll"])}.get(physics, "tvdlf")
    walls = "tube" if start == "tube" else rng.choice(["periodic", "mixed"]) if start == "waves" else "periodic"
    losses = physics in ("hd", "ffhd", "ffhd_htc") and start != "tube" and rng.random() < 0.3
    steps = rng.randint(4, 20) if nbytes == 4 else rng.randint(2, 5)
    return _case(physics=physics, start=start, limiter=limiter, flux=flux, rk=rk, bytes=nbytes, bx=bx, by=by, bz=bz,
                 walls=walls, steps=steps, host_dt=rng.random() < 0.25, losses=losses,
                 sums_every=rng.choice([0, 0, 5]),
                 eos="synge" if physics == "srhd" and rng.random() < 0.3 else "ideal")


# ------------------------------------------------------------------------------------ inputs
def _grid(nb):
    """Cell-centre coordinates in [0, 1]^3, shaped to broadcast as (z, y, x)."""
    ax = [(torch.arange(16 * n, device="cuda", dtype=torch.float64) + 0.5) / (16 * n) for n in nb]
    return ax[0].view(1, 1, -1), ax[1].view(1, -1, 1), ax[2].view(-1, 1, 1)


def _start(kind, physics, nb, rnd, noise):
    """Primitive fields (variable, z, y, x) in FP64. rnd: a numpy RandomState; noise: a torch
    generator for per-cell noise."""
    x, y, z = _grid(nb)
    shape = (16 * nb[2], 16 * nb[1], 16 * nb[0])
    p = torch.zeros((NV[physics],) + shape, device="cuda", dtype=torch.float64)
    ph = rnd.uniform(0.0, TP, 64)

    def per_cell():
        return 2.0 * torch.rand(shape, device="cuda", dtype=torch.float64, generator=noise) - 1.0

    if kind == "tube":            # the Sod states either side of a plane, weakly disturbed
        left = x < rnd.uniform(0.4, 0.6)
        p[0] = torch.where(left, 1.0, 0.125)
        p[4] = torch.where(left, 1.0, 0.1)
        p[0] *= 1.0 + 0.02 * torch.sin(TP * y + ph[0]) * torch.cos(TP * z + ph[1])
        p[2] = 0.05 * torch.sin(TP * (y + z) + ph[2])
    elif kind == "shear":         # double shear layer with a seeded disturbance
        w = 0.02
        inner = 0.5 * (torch.tanh((y - 0.25) / w) - torch.tanh((y - 0.75) / w))
        p[0] = 1.0 + inner
        p[1] = 0.5 * (1.0 - 2.0 * inner)
        p[2] = 0.01 * torch.sin(2 * TP * x + ph[0]) * (1.0 + 0.1 * torch.sin(TP * z + ph[1]))
        p[1:4] += 0.005 * torch.stack([per_cell() for _ in range(3)])
        p[4] = 2.5
    elif kind == "vortex":        # Orszag-Tang-like fields with 1% velocity noise
        b0 = math.sqrt(2.0 / 3.0)
        cz = torch.cos(TP * z + ph[0])
        p[0] = 4.0
        p[1] = -torch.sin(TP * y + ph[1]) * cz
        p[2] = torch.sin(TP * x + ph[2]) * cz
        p[4] = 1.0
        p[5] = -b0 * torch.sin(TP * y + ph[3]) * cz
        p[6] = b0 * torch.sin(2 * TP * x + ph[4]) * cz
        p[1:4] += 0.01 * torch.stack([per_cell() for _ in range(3)])
    elif kind == "waves":         # a few smooth modes in every variable
        for v in range(NV[physics]):
            for m in range(3):
                k = rnd.randint(1, 4, 3)
                p[v] += rnd.uniform(-0.5, 0.5) * torch.sin(TP * (k[0] * x + k[1] * y + k[2] * z) + ph[3 * v + m])
        p[0] = 1.0 + 0.3 * torch.tanh(p[0])
        p[4] = 1.0 + 0.3 * torch.tanh(p[4])
        if physics == "mhd":
            p[8] *= 0.05
    elif kind == "blast":         # a hot sphere, off centre, in a uniform (magnetised) gas
        # density and energy are the same for every seed, so that the estimator refines the
        # same blocks; the seed sets the flow (and the field's direction) beneath them
        longest = float(max(nb))
        r2 = sum(((q - ci) * n / longest) ** 2 for q, ci, n in zip((x, y, z), (0.47, 0.53, 0.45), nb))
        p[0] = 1.0
        k = rnd.randint(1, 3, (3, 3))
        for i in range(3):
            p[1 + i] = 0.15 * torch.sin(TP * (k[i, 0] * x + k[i, 1] * y + k[i, 2] * z) + ph[i])
        p[4] = torch.where(r2 < 0.12 ** 2, 10.0, 0.1) - (GAMMA[physics] - 1.0) * 0.5 * (p[1:4] ** 2).sum(0)
        if physics == "mhd":
            p[5] = 0.3 * math.cos(ph[4])
            p[6] = 0.3 * math.sin(ph[4])
    elif kind == "shell":         # a relativistic spherical shell moving outwards
        c = rnd.uniform(0.0, 1.0, 3)
        rad, rho, lor = rnd.uniform(0.2, 0.35), rnd.uniform(1.0, 10.0), rnd.uniform(1.0, 6.0)
        d = [q - ci for q, ci in zip((x, y, z), c)]
        d = [q - torch.floor(q + 0.5) for q in d]
        r = torch.sqrt(d[0] ** 2 + d[1] ** 2 + d[2] ** 2)
        w = torch.exp(-((r - rad) * 16 * min(nb)) ** 2 / 8.0)
        p[0] = 1.0 + (rho - 1.0) * w
        u = w * math.sqrt(lor * lor - 1.0) / r.clamp_min(1e-9)
        for i in range(3):
            p[1 + i] = u * d[i]
        p[4] = 1.0
    elif kind == "loop":          # flow and temperature waves along a curved frozen field
        th = 0.7 * torch.sin(TP * x + ph[0]) + 0.5 * torch.cos(TP * (y + z) + ph[1])
        p[0] = 1.0 + 0.3 * torch.sin(TP * (x + 2 * y) + ph[2]) * torch.cos(TP * z + ph[3])
        p[1] = 0.4 * torch.cos(TP * (x - y) + ph[4])
        p[2] = 1.0 + 0.4 * torch.sin(TP * (y + z) + ph[5]) * torch.cos(TP * x + ph[6])
        b = NV[physics] - 3
        if b == 4:
            p[3] = 0.01 * torch.sin(TP * (x + y - z) + ph[7])
        p[b] = torch.cos(th) * torch.cos(0.3 * th)
        p[b + 1] = torch.sin(th) * torch.cos(0.3 * th)
        p[b + 2] = torch.sin(0.3 * th)
    else:
        raise ValueError(kind)
    return p


def _morton(nb):
    """Block coordinates (x, y, z) in Z-order, the library's order of the blocks of a mesh."""
    at = [(i, j, k) for k in range(nb[2]) for j in range(nb[1]) for i in range(nb[0])]
    return sorted(at, key=lambda c: sum(((c[d] >> b) & 1) << (3 * b + d) for b in range(5) for d in range(3)))


def _to_blocks(f, nb):
    """(variable, z, y, x) -> (block, variable, 16, 16, 16) in Z-order."""
    v = f.shape[0]
    b = f.reshape(v, nb[2], 16, nb[1], 16, nb[0], 16).permute(1, 3, 5, 0, 2, 4, 6).reshape(-1, v, 16, 16, 16)
    at = torch.tensor([(k * nb[1] + j) * nb[0] + i for i, j, k in _morton(nb)], device=f.device)
    return b[at]


def _solves(case):
    """The block counts of the case's solves (a batch's solves are cubes)."""
    if case["kind"] == "batch":
        return [(int(s),) * 3 for s in case["sizes"].split(",")]
    return [(case["bx"], case["by"], case["bz"])]


def _fields(case, seed, i, nb):
    s = (seed * 1000003 + 7919 * i) % (1 << 31)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(s)
    return _start(case["start"], case["physics"], nb, np.random.RandomState(s), gen)


def _config(case, nb):
    extra = {}
    if case["levels"] > 1:
        extra = dict(max_level=case["levels"], refine_vars=(0, 4), refine_weights=(0.5, 0.5), refine_tol=0.2)
    return agile.make_config(physics=case["physics"], limiter=case["limiter"], flux=case["flux"], rk=case["rk"],
                             real_bytes=case["bytes"], gamma=GAMMA[case["physics"]], base_blocks=nb,
                             bc=WALLS[case["walls"]], eos=case["eos"],
                             htc_kappa0=KAPPA0 if case["physics"] == "ffhd_htc" else 0.0, **extra)


def _table():
    return workloads.skew_normal_cooling(n=128, peak=1.0)


def _dp(t):
    return C.cast(t.data_ptr(), C.POINTER(C.c_double))


# ------------------------------------------------------------------------------------ passes
def prepare(case, seed):
    nbs = _solves(case)
    prims, outs = [], []
    joins = len(nbs) // 2
    for i, nb in enumerate(nbs + (nbs[joins:joins + 1] if case["kind"] == "batch" else [])):
        blocks = _to_blocks(_fields(case, seed, i, nb), nb)
        host = torch.empty(blocks.shape, dtype=torch.float64, pin_memory=True)
        host.copy_(blocks)
        prims.append(host)
        if case["kind"] != "amr" and i < len(nbs):
            outs.append(torch.empty_like(host, pin_memory=True))
    state = {"case": case, "prims": prims, "outs": outs, "cfgs": [_config(case, nb) for nb in nbs]}
    if case["kind"] == "mesh":
        state["mesh"] = agile.Mesh(state["cfgs"][0])
        if case["losses"]:
            state["mesh"].set_cooling(*_table())
    elif case["kind"] == "batch":
        state["batch"] = agile.Batch(state["cfgs"])
        state["slots"] = list(range(len(nbs)))
    else:
        # room for every leaf the refined mesh can have in this case
        most = nbs[0][0] * nbs[0][1] * nbs[0][2] * (64 if case["levels"] > 3 else 40)
        state["room"] = torch.empty((most, NV[case["physics"]], 16, 16, 16), dtype=torch.float64, pin_memory=True)
    return state


def _get(call, handle, out, *which):
    st = call(handle, *which, None, None, _dp(out))
    if st != 0:
        raise RuntimeError("reading the state failed with status %d" % st)
    return out


def _advance(mesh, case):
    sums = []
    for n in range(case["steps"]):
        if case["host_dt"]:
            mesh.step(mesh.cfl_dt())
        else:
            mesh.step(0.0)
        if case["sums_every"] and (n + 1) % case["sums_every"] == 0:
            sums.append(mesh.conserved_sums())
    return sums


def run(state):
    case, lib = state["case"], agile.load()
    if case["kind"] == "mesh":
        mesh = state["mesh"]
        mesh.set_state_prims(state["prims"][0].numpy())
        sums = _advance(mesh, case)
        out = [_get(lib.agile_get_state, mesh.ptr, state["outs"][0])]
        return out + ([np.stack(sums)] if sums else [])
    if case["kind"] == "amr":
        # a refined solve from its creation on: the estimator refines around the blast
        mesh = agile.Mesh(state["cfgs"][0])
        mesh.set_state_prims(state["prims"][0].numpy())
        for _ in range(case["levels"] - 1):
            mesh.regrid()
        _advance(mesh, case)
        n = mesh.layout()[0]
        if n > state["room"].shape[0]:
            raise RuntimeError("more leaves than expected: %d" % n)
        out = _get(lib.agile_get_state, mesh.ptr, state["room"][:n])
        mesh.close()
        return [out]
    batch, slots, half = state["batch"], state["slots"], len(state["cfgs"]) // 2
    for i, s in enumerate(slots):
        batch.set_state_prims(s, state["prims"][i].numpy())
    for n in range(case["steps"]):
        if n == case["steps"] // 2:
            batch.detach(slots[half])
            slots[half] = batch.attach(state["cfgs"][half])
            batch.set_state_prims(slots[half], state["prims"][-1].numpy())
        batch.step()
    return [_get(lib.agile_batch_get_state, batch.ptr, out, s) for out, s in zip(state["outs"], slots)]


def work(case):
    """State in and out once over the host link (FP64), and per cell and stage the stage input
    read, the output written and U^n read again in the combining stages."""
    cells = sum(a * b * c for a, b, c in _solves(case)) * 4096.0
    if case["kind"] == "amr":        # about what the refinement around the blast makes of it
        cells *= 12.0 if case["levels"] > 3 else 8.0
    nv, nt, rk = NV[case["physics"]], NT[case["physics"]], case["rk"]
    per_step = cells * case["bytes"] * (nt * 2 * rk + nv * (rk - 1))
    return {"bytes": case["steps"] * per_step + 2 * 8.0 * nv * cells,
            "flops": case["steps"] * rk * cells * FLOPS[case["physics"]]}


def tolerance(case):
    # FP64: against plain FP64 (exact below) a pass is 1e-16 to 3e-16 off, FP32: 7e-8 to 8e-7, at
    # steep fronts (where rounding decides which way a limiter goes) up to 1.6e-6
    if case["bytes"] == 8:           # relativistic shells, whose recovery iterates: up to 1.4e-15
        return {"rel": 1e-14 if case["start"] == "shell" else 4e-15, "max": 1e-11}
    if case["start"] in ("tube", "blast", "shell"):
        return {"rel": 8e-6, "max": 2e-3}
    return {"rel": 4e-6, "max": 4e-4}


# ------------------------------------------------------------------- the same in plain FP64
# An independent statement of the scheme on a uniform grid: fields (variable, z, y, x), the
# six boundaries by padding along one axis at a time, every face flux from two PLM states.
def _axis(d):
    return 3 - d                          # tensor axis of direction d (0 = x)


def _pad(f, d, walls, flips):
    ax, n = _axis(d), f.shape[_axis(d)]
    kinds = WALLS[walls][2 * d:2 * d + 2]
    ends = []
    for s, kind in enumerate(kinds):
        if kind == "periodic":
            g = f.narrow(ax, n - 2, 2) if s == 0 else f.narrow(ax, 0, 2)
        elif kind == "outflow":
            one = f.narrow(ax, 0 if s == 0 else n - 1, 1)
            g = torch.cat([one, one], ax)
        else:
            g = f.narrow(ax, 0 if s == 0 else n - 2, 2).flip(ax).clone()
            for v in flips:
                g[v + d].neg_()
        ends.append(g)
    return torch.cat([ends[0], f, ends[1]], ax)


def _half(a, b, limiter):
    same = a * b > 0
    if limiter == "minmod":
        m = torch.minimum(a.abs(), b.abs()) * torch.sign(a) * 0.5
    else:
        m = a * b / torch.where(same, a + b, torch.ones_like(a))
    return torch.where(same, m, torch.zeros_like(m))


class _Gas:
    def __init__(self, case):
        self.case, self.g, self.kind = case, GAMMA[case["physics"]], case["physics"]
        self.flips = {"hd": (1,), "srhd": (1,), "mhd": (1, 5), "ffhd": (3,), "ffhd_htc": (4,)}[self.kind]
        self.vec = self.kind in ("hd", "mhd", "srhd")
        self.b = NV[self.kind] - 3        # first field component (ffhd)
        self.ch = 0.0

    def cons(self, p):
        u, g = p.clone(), self.g
        if self.kind == "srhd":
            lor = (1 + (p[1:4] ** 2).sum(0)).sqrt()
            w = lor * lor * (p[0] + g / (g - 1) * p[4])
            u[0] = lor * p[0]
            u[1:4] = w / lor * p[1:4]
            u[4] = w - p[4] - u[0]
        elif self.vec:
            u[1:4] = p[0] * p[1:4]
            u[4] = p[4] / (g - 1) + 0.5 * p[0] * (p[1:4] ** 2).sum(0)
            if self.kind == "mhd":
                u[4] += 0.5 * (p[5:8] ** 2).sum(0)
        else:
            u[1] = p[0] * p[1]
            u[2] = p[2] / (g - 1) + 0.5 * p[0] * p[1] ** 2
        return u

    def prims(self, u):
        p, g = u.clone(), self.g
        if self.kind == "srhd":
            # root of the energy equation in the pressure, by bisection to a narrow bracket and
            # Newton steps from there
            m2, e = (u[1:4] ** 2).sum(0), u[4] + u[0]

            def off(pr):
                w = e + pr
                v2 = m2 / (w * w)
                lor = 1 / (1 - v2).sqrt()
                rho = u[0] / lor
                eps = (w * (1 - v2) - rho - pr) / rho          # specific internal energy
                cs2 = g * (g - 1) * eps / (1 + g * eps)
                return (g - 1) * rho * eps - pr, v2 * cs2 - 1, lor, rho
            lo = (m2.sqrt() - e).clamp_min(0.0)
            hi = (g - 1) * e
            for _ in range(30):
                mid = 0.5 * (lo + hi)
                f = off(mid)[0]
                up = (f > 0) | torch.isnan(f)
                lo, hi = torch.where(up, mid, lo), torch.where(up, hi, mid)
            pr = 0.5 * (lo + hi)
            for _ in range(4):
                f, df, _, _ = off(pr)
                pr = pr - f / df
            _, _, lor, rho = off(pr)
            p[0], p[4] = rho, pr
            p[1:4] = u[1:4] * lor / (e + pr)
        elif self.vec:
            p[1:4] = u[1:4] / u[0]
            ek = 0.5 * (u[1:4] * p[1:4]).sum(0)
            if self.kind == "mhd":
                ek += 0.5 * (u[5:8] ** 2).sum(0)
            p[4] = (g - 1) * (u[4] - ek)
        else:
            p[1] = u[1] / u[0]
            p[2] = (g - 1) * (u[2] - 0.5 * u[1] * p[1])
        return p

    def speeds(self, p, d):
        """Smallest and largest characteristic speed along d."""
        g = self.g
        if self.kind == "hd":
            c = (g * p[4] / p[0]).sqrt()
            return p[1 + d] - c, p[1 + d] + c
        if self.kind == "mhd":
            a2, b2, bd2 = g * p[4] / p[0], (p[5:8] ** 2).sum(0) / p[0], p[5 + d] ** 2 / p[0]
            s = a2 + b2
            c = (0.5 * (s + (s * s - 4 * a2 * bd2).clamp_min(0).sqrt())).sqrt()
            return p[1 + d] - c, p[1 + d] + c
        if self.kind == "srhd":
            lor2 = 1 + (p[1:4] ** 2).sum(0)
            v2, v = 1 - 1 / lor2, p[1 + d] / lor2.sqrt()
            cs2 = g * p[4] / (p[0] + g / (g - 1) * p[4])
            root = (cs2 * (1 - v2) * (1 - v2 * cs2 - v * v * (1 - cs2)).clamp_min(0)).sqrt()
            return (v * (1 - cs2) - root) / (1 - v2 * cs2), (v * (1 - cs2) + root) / (1 - v2 * cs2)
        c, bd = (g * p[2] / p[0]).sqrt(), p[self.b + d]
        return p[1] * bd - c * bd.abs(), p[1] * bd + c * bd.abs()

    def flux(self, p, u, d):
        f = torch.zeros_like(p)
        if self.kind == "srhd":
            v = p[1 + d] / (1 + (p[1:4] ** 2).sum(0)).sqrt()
            f[0:4] = u[0:4] * v
            f[1 + d] += p[4]
            f[4] = u[1 + d] - u[0] * v
        elif self.kind == "hd":
            f[0:4] = u[0:4] * p[1 + d]
            f[1 + d] += p[4]
            f[4] = (u[4] + p[4]) * p[1 + d]
        elif self.kind == "mhd":
            v, b = p[1 + d], p[5 + d]
            pt = p[4] + 0.5 * (p[5:8] ** 2).sum(0)
            f[0] = u[0] * v
            f[1:4] = u[1:4] * v - p[5:8] * b
            f[1 + d] += pt
            f[4] = (u[4] + pt) * v - b * (p[1:4] * p[5:8]).sum(0)
            f[5:8] = v * p[5:8] - b * p[1:4]
            f[5 + d] = p[8]
            f[8] = self.ch ** 2 * b
        else:
            b = p[self.b + d]
            f[0] = u[0] * p[1] * b
            f[1] = (u[1] * p[1] + p[2]) * b
            f[2] = (u[2] + p[2]) * p[1] * b
            if self.kind == "ffhd_htc":
                f[2] -= p[3] * b
            f[self.b + d] = b
        return f

    def face(self, pl, pr, d):
        if self.kind == "mhd":
            bl, br, sl, sr = pl[5 + d].clone(), pr[5 + d].clone(), pl[8].clone(), pr[8].clone()
            for q in (pl, pr):
                q[5 + d] = 0.5 * (bl + br) - 0.5 * (sr - sl) / self.ch
                q[8] = 0.5 * (sl + sr) - 0.5 * self.ch * (br - bl)
        if not self.vec:
            m = 0.5 * (pl[self.b + d] + pr[self.b + d])
            pl[self.b + d] = m
            pr[self.b + d] = m
        ul, ur = self.cons(pl), self.cons(pr)
        fl, fr = self.flux(pl, ul, d), self.flux(pr, ur, d)
        (al, bl), (ar, br) = self.speeds(pl, d), self.speeds(pr, d)
        name = self.case["flux"]
        if name == "tvdlf":
            c = torch.maximum(torch.maximum(al.abs(), bl.abs()), torch.maximum(ar.abs(), br.abs()))
            f = 0.5 * (fl + fr) - 0.5 * c * (ur - ul)
            if not self.vec:
                f[self.b:] = fl[self.b:]
                if self.kind == "ffhd_htc":
                    f[3] = 0
            return f
        lo, hi = torch.minimum(al, ar), torch.maximum(bl, br)
        if name == "hll":
            lo, hi = lo.clamp_max(0), hi.clamp_min(0)
            return (hi * fl - lo * fr + lo * hi * (ur - ul)) / (hi - lo)
        # HLLC: the contact restored between the outer waves
        ml, mr = pl[0] * (lo - pl[1 + d]), pr[0] * (hi - pr[1 + d])
        sc = (pr[4] - pl[4] + ml * pl[1 + d] - mr * pr[1 + d]) / (ml - mr)

        def star(p, u, m, s):
            r = m / (s - sc)
            q = torch.empty_like(u)
            q[0] = r
            q[1:4] = r * p[1:4]
            q[1 + d] = r * sc
            q[4] = r * (u[4] / p[0] + (sc - p[1 + d]) * (sc + p[4] / m))
            return q
        f = torch.where(sc >= 0, fl + lo * (star(pl, ul, ml, lo) - ul), fr + hi * (star(pr, ur, mr, hi) - ur))
        return torch.where(lo >= 0, fl, torch.where(hi <= 0, fr, f))

    def rate(self, u, dx, dt):
        p = self.prims(u)
        out = torch.zeros_like(u)
        grad = 0.0
        for d in range(3):
            ax = _axis(d)
            q = _pad(p, d, self.case["walls"], self.flips)
            n = p.shape[ax]
            dq = q.narrow(ax, 1, n + 3) - q.narrow(ax, 0, n + 3)
            h = _half(dq.narrow(ax, 0, n + 2), dq.narrow(ax, 1, n + 2), self.case["limiter"])
            if not self.vec:
                h[self.b:] = 0
            mid = q.narrow(ax, 1, n + 2)
            f = self.face((mid + h).narrow(ax, 0, n + 1), (mid - h).narrow(ax, 1, n + 1), d)
            out -= (f.narrow(ax, 1, n) - f.narrow(ax, 0, n)) / dx[d]
            if self.kind == "ffhd_htc":
                t = q[2] / q[0]
                grad = grad + p[self.b + d] * (t.narrow(ax - 1, 3, n) - t.narrow(ax - 1, 1, n)) / (2 * dx[d])
        if not self.vec:
            out[1] -= p[2] * out[self.b:].sum(0)
            out[self.b:] = 0
            if self.kind == "ffhd_htc":
                out[3] = (KAPPA0 * (p[2] / p[0]) ** 2.5 * grad - p[3]) / (4 * dt)
        return out


def _evolve(case, prim, nb):
    gas, dx = _Gas(case), [1.0 / (16 * n) for n in nb]
    u = gas.cons(prim)
    sums = []
    for n in range(case["steps"]):
        p = gas.prims(u)
        s = [torch.maximum(lo.abs(), hi.abs()) for lo, hi in (gas.speeds(p, d) for d in range(3))]
        dt = 0.4 / float((s[0] / dx[0] + s[1] / dx[1] + s[2] / dx[2]).max())
        gas.ch = float(max(q.max() for q in s))
        fade = math.exp(-0.5 * dt * gas.ch * 0.5 / min(dx))
        if case["physics"] == "mhd":
            u[8] *= fade
        u0 = u.clone()
        for a, b in ((0, 1), (0.5, 0.5)) if case["rk"] == 2 else ((0, 1), (0.75, 0.25), (1 / 3, 2 / 3)):
            u = a * u0 + b * (u + dt * gas.rate(u, dx, dt))
        if case["physics"] == "mhd":
            u[8] *= fade
        if case["sums_every"] and (n + 1) % case["sums_every"] == 0:
            sums.append(u.flatten(1).sum(1) * (dx[0] * dx[1] * dx[2]))
    return [_to_blocks(u, nb)] + ([torch.stack(sums)] if sums else [])


def exact(case, seed):
    cells = sum(a * b * c for a, b, c in _solves(case)) * 4096
    if (case["kind"] == "amr" or case["losses"] or case["eos"] != "ideal"
            or cells * case["steps"] * case["rk"] * NV[case["physics"]] > 6e9):
        return None
    out = []
    for i, nb in enumerate(_solves(case)):
        joined = case["kind"] == "batch" and i == len(_solves(case)) // 2
        c = dict(case, steps=case["steps"] - case["steps"] // 2) if joined else case
        prim = _fields(case, seed, len(_solves(case)) if joined else i, nb)
        got = _evolve(c, prim, nb)
        out += got if case["kind"] == "mesh" else got[:1]
    return out
