"""Stage launches of few blocks cut the blocks along z (the stage kernel's work items are 16, 8,
4, 2 or 1 planes, chosen from the number of blocks in the launch): a small solve, alone cut into
single planes, gives the same bits in batches whose launches take larger items and whole
blocks, for every physics module and precision, at walls in z and on refined meshes."""
import numpy as np
import pytest

from paper_2607_19277_gb300 import agile, workloads as W

pytestmark = pytest.mark.gpu
PER, OUT, REF = "periodic", "outflow", "reflect"


def _loop(x, y, z):
    p = np.zeros((7,) + np.shape(x))
    th = 0.7 * np.sin(2 * np.pi * (x + z))
    p[0] = 1.0 + 0.3 * np.sin(2 * np.pi * (y - z))
    p[1] = 0.4 * np.cos(2 * np.pi * z)
    p[2] = 1.0 + 0.3 * np.cos(2 * np.pi * x)
    p[4], p[5], p[6] = np.cos(th) * np.cos(0.3 * th), np.sin(th) * np.cos(0.3 * th), np.sin(0.3 * th)
    return p


def _ic(physics):
    if physics == "srhd":   # (prolonging stronger shear leaves states without primitives, in the oracle too)
        return W.srhd_shells(7, 48, n_shells=1, smooth=True, width=4, lorentz_max=2, p_amb=1.0)
    return _loop if physics == "ffhd_htc" else W.random_smooth(agile.NVAR[agile.PHYSICS[physics]], 5, physics)


def _run(cfgs, physics, flags, steps=2):
    b = agile.Batch(cfgs)
    for i in range(len(cfgs)):
        b.set_state(i, _ic(physics))
    if flags is not None:
        b.regrid_flags(0, flags)
    for _ in range(steps):
        b.step()
    lev, ijk, cons = b.get_state(0)
    b.close()
    return lev, ijk, cons


@pytest.mark.parametrize("physics,rb,flux,limiter,bc,refine", [
    ("hd", 8, "hll", "minmod", (PER,) * 6, False),
    ("hd", 4, "hllc", "vanleer", (OUT, REF, PER, PER, REF, OUT), False),
    ("mhd", 8, "tvdlf", "vanleer", (OUT, OUT, PER, PER, REF, REF), False),
    ("mhd", 4, "hll", "vanleer", (PER,) * 6, False),
    ("srhd", 8, "tvdlf", "minmod", (PER, PER, OUT, OUT, OUT, REF), False),
    ("srhd", 4, "tvdlf", "vanleer", (PER,) * 6, False),
    ("ffhd_htc", 4, "tvdlf", "vanleer", (PER, PER, PER, PER, REF, OUT), False),
    ("hd", 4, "tvdlf", "minmod", (OUT,) * 6, True),
    ("mhd", 8, "hll", "minmod", (PER,) * 6, True),
    ("srhd", 4, "tvdlf", "vanleer", (PER,) * 6, True),
])
def test_items_give_the_same_bits(physics, rb, flux, limiter, bc, refine):
    common = dict(physics=physics, limiter=limiter, flux=flux, rk=2, real_bytes=rb,
                  htc_kappa0=1e-3 if physics == "ffhd_htc" else 0.0)
    cfg = agile.make_config(base_blocks=(2, 1, 3), bc=bc, max_level=2 if refine else 1, **common)
    flags = None
    if refine:
        flags = np.zeros(6, dtype=np.int32)
        flags[[0, 3]] = 1
    alone = _run([cfg], physics, flags)
    for nx, ny, nz in ((4, 4, 2), (5, 4, 4), (6, 6, 4), (8, 6, 8)):     # blocks beside the solve
        mixed = _run([cfg, agile.make_config(base_blocks=(nx, ny, nz), **common)], physics, flags)
        for a, m in zip(alone, mixed):
            assert np.array_equal(a, m), (nx, ny, nz)
