"""Blocks whose faces take the coarse-fine flux correction get their CFL maxima (and, for MHD, the
second GLM half) in passes over them alone, every other block in the last stage's stores: the
CFL step after a step on a three-level mesh equals the one reduced afresh from the same state,
also where the fastest cell lies in such a block, on an edge of two corrected faces."""
import numpy as np
import pytest

from paper_2607_19277_gb300 import agile, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("physics,rb", [("hd", 8), ("hd", 4), ("mhd", 8), ("mhd", 4)])
@pytest.mark.parametrize("hot", ["corrected", "other"])
def test_cfl_after_a_step(physics, rb, hot):
    nv = agile.NVAR[agile.PHYSICS[physics]]
    smooth = W.random_smooth(nv, 9, physics)
    # base 3 x 2 x 2; blocks (1, 0, 0) and (0, 1, 0) refine, (0, 0, 0) keeps two corrected faces
    at = (0.31, 0.48, 0.2) if hot == "corrected" else (0.95, 0.95, 0.95)

    def ic(x, y, z):
        p = smooth(x, y, z)
        r2 = (x - at[0]) ** 2 + (y - at[1]) ** 2 + (z - at[2]) ** 2
        p[4] = p[4] + 30.0 * np.exp(-r2 / 0.01)
        return p

    m = agile.Mesh(agile.make_config(physics=physics, limiter="minmod", flux="hll", rk=2, real_bytes=rb,
                                     base_blocks=(3, 2, 2), bc=("outflow",) * 6, max_level=3))
    m.set_state(ic)
    lev, ijk, _ = m.get_state()
    flags = np.array([1 if tuple(c) in ((1, 0, 0), (0, 1, 0)) else 0 for c in ijk], dtype=np.int32)
    assert m.regrid_flags(flags, init=True)[0] == 2
    lev, ijk, _ = m.get_state()
    flags = np.zeros(len(lev), dtype=np.int32)
    flags[np.flatnonzero(lev == 2)[3]] = 1
    m.regrid_flags(flags, init=True)
    lev = m.get_state()[0]
    assert set(lev) == {1, 2, 3}
    for _ in range(2):
        m.step(0.0)
    a = m.max_speeds()
    m.set_state_blocks(m.get_state()[2])
    b = m.max_speeds()
    m.close()
    # the same maxima of the same cells; the two kernels may contract products differently
    ulp = 2.0 ** -52 if rb == 8 else 2.0 ** -22
    assert a == pytest.approx(b, rel=4 * ulp)
