"""Stage launches of few blocks cut the blocks along z (the stage kernel's work items are 16, 8,
4, 2 or 1 planes, chosen from the number of blocks in the launch): a small solve, alone cut into
single planes, gives the same bits in batches whose launches take larger items and whole
blocks, for every physics module and precision, at walls in z and on refined meshes."""
import numpy as np
import pytest

from paper_2607_19277_gb300 import agile, workloads as W
from parity_util import side_by_side, stage_ic

pytestmark = pytest.mark.gpu
PER, OUT, REF = "periodic", "outflow", "reflect"


def _ic(physics):
    if physics == "srhd":   # (prolonging stronger shear leaves states without primitives, in the oracle too)
        return W.srhd_shells(7, 48, n_shells=1, smooth=True, width=4, lorentz_max=2, p_amb=1.0)
    return stage_ic(physics)


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
    ("synge", 8, "tvdlf", "minmod", (PER, PER, OUT, OUT, OUT, REF), False),
    ("synge", 4, "tvdlf", "vanleer", (PER,) * 6, False),
    ("ffhd", 8, "tvdlf", "minmod", (PER, PER, PER, PER, OUT, REF), False),
    ("ffhd", 4, "tvdlf", "vanleer", (PER, PER, PER, PER, REF, OUT), False),
    ("ffhd_htc", 8, "tvdlf", "vanleer", (PER,) * 6, False),
    ("ffhd_htc", 4, "tvdlf", "vanleer", (PER, PER, PER, PER, REF, OUT), False),
    ("hd", 4, "tvdlf", "minmod", (OUT,) * 6, True),
    ("mhd", 8, "hll", "minmod", (PER,) * 6, True),
    ("srhd", 4, "tvdlf", "vanleer", (PER,) * 6, True),
])
def test_items_give_the_same_bits(physics, rb, flux, limiter, bc, refine):
    eos = "synge" if physics == "synge" else "ideal"
    physics = "srhd" if physics == "synge" else physics
    common = dict(physics=physics, limiter=limiter, flux=flux, rk=2, real_bytes=rb, eos=eos,
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


@pytest.mark.parametrize("rb", [8, 4])
def test_items_give_the_same_bits_with_resistivity(rb):
    alone = side_by_side((1, 1, 1), rb)
    for reps in ((3, 3, 2), (3, 4, 5), (4, 4, 5), (4, 6, 4)):           # 108 to 576 blocks
        assert np.array_equal(alone, side_by_side(reps, rb)), reps
