"""Stage launches of some tens to some thousand blocks may leave the first blocks whole and cut the
others into items of a planes and one of the rest: a small solve at the end of a batch, where the
cut blocks are, gives the same bits as alone (equal items), at numbers of blocks that give a = 2
to 13 planes, and none, one or more rounds of whole blocks first."""
import numpy as np
import pytest

from paper_2607_19277_gb300 import agile
from parity_util import side_by_side, stage_ic

pytestmark = pytest.mark.gpu
PER, OUT, REF = "periodic", "outflow", "reflect"


def _last(cfgs, physics):
    b = agile.Batch(cfgs)
    for i in range(len(cfgs)):
        b.set_state(i, stage_ic(physics))
    for _ in range(2):
        b.step()
    lev, ijk, cons = b.get_state(len(cfgs) - 1)
    b.close()
    return lev, ijk, cons


@pytest.mark.parametrize("physics,rb,flux,limiter,bc", [
    ("hd", 8, "hllc", "minmod", (PER,) * 6),
    ("mhd", 8, "hll", "vanleer", (OUT, REF, PER, PER, REF, OUT)),
    ("srhd", 8, "tvdlf", "vanleer", (PER,) * 6),
    ("hd", 4, "hll", "vanleer", (OUT, OUT, PER, PER, REF, REF)),
    ("mhd", 4, "tvdlf", "minmod", (PER, PER, OUT, OUT, OUT, REF)),
    ("srhd", 4, "tvdlf", "minmod", (PER,) * 6),
    ("synge", 8, "tvdlf", "minmod", (PER,) * 6),
    ("synge", 4, "tvdlf", "vanleer", (PER,) * 6),
    ("ffhd", 8, "tvdlf", "vanleer", (PER, PER, PER, PER, REF, OUT)),
    ("ffhd", 4, "tvdlf", "minmod", (PER,) * 6),
    ("ffhd_htc", 8, "tvdlf", "minmod", (PER,) * 6),
    ("ffhd_htc", 4, "tvdlf", "vanleer", (PER,) * 6),
])
def test_uneven_items_give_the_same_bits(physics, rb, flux, limiter, bc):
    eos = "synge" if physics == "synge" else "ideal"
    physics = "srhd" if physics == "synge" else physics
    common = dict(physics=physics, limiter=limiter, flux=flux, rk=2, real_bytes=rb, eos=eos,
                  htc_kappa0=1e-3 if physics == "ffhd_htc" else 0.0)
    cfg = agile.make_config(base_blocks=(2, 1, 3), bc=bc, **common)
    alone = _last([cfg], physics)
    for nblk in (42, 60, 80, 90, 120, 210, 340, 400, 512, 1250):
        beside = agile.make_config(base_blocks=((nblk - 6) // 2, 2, 1), **common)
        for a, m in zip(alone, _last([beside, cfg], physics)):
            assert np.array_equal(a, m), nblk


@pytest.mark.parametrize("rb", [8, 4])
def test_uneven_items_give_the_same_bits_with_resistivity(rb):
    """Resistive MHD, which batches refuse: a periodic mesh and copies of it side by side."""
    alone = side_by_side((1, 1, 1), rb)
    for reps in ((7, 1, 1), (2, 5, 1), (5, 4, 1), (5, 17, 1), (10, 4, 5)):     # 42 to 1200 blocks
        assert np.array_equal(alone, side_by_side(reps, rb)), reps
