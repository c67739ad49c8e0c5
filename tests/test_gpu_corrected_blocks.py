"""Blocks whose faces take the coarse-fine flux correction get their CFL maxima (and, for MHD, the
second GLM half) in passes over them alone, every other block in the last stage's stores: the
CFL step after a step on a three-level mesh equals the one reduced afresh from the same state,
also where the fastest cell lies in such a block, on an edge of two corrected faces; and psi, which
the second half multiplies, agrees with the oracle's in the corrected blocks as in the others."""
import numpy as np
import pytest

from paper_2607_19277_gb300 import agile, workloads as W
from parity_util import TOL_FP32, TOL_FP64, force_refine, gpu_mesh, oracle_solver

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


@pytest.mark.parametrize("rb,tol", [(8, TOL_FP64), (4, TOL_FP32)])
def test_second_glm_half(rb, tol):
    spec = dict(physics="mhd", limiter="minmod", flux="hll", rk=2, base_blocks=(3, 2, 2), bc=("outflow",) * 6,
                max_level=3)
    ic = W.random_smooth(9, 9, "mhd")
    o, m = oracle_solver(spec), gpu_mesh(spec, rb)
    o.set_state(ic)
    m.set_state(ic)
    force_refine(o, m, {(1, 1, 0, 0), (1, 0, 1, 0)})
    force_refine(o, m, {(2, 2, 1, 1)})
    m.set_state_blocks(o.get_state()[2])
    for _ in range(2):
        dt = o.cfl_dt()
        o.step(dt)
        m.step(dt)
    lev, ijk, g = m.get_state()
    r = o.get_state()[2]
    m.close()
    keys = {(l, *c) for l, c in zip(lev.tolist(), ijk.tolist())}
    fine = {(l - 1, x >> 1, y >> 1, z >> 1) for l, x, y, z in keys if l > 1}
    # a block is corrected where the block beside it, at its own level, is refined
    corrected = np.array([any((l, *np.add((x, y, z), d)) in fine for d in
                              ((1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)))
                          for l, (x, y, z) in zip(lev.tolist(), ijk.tolist())])
    assert corrected.sum() >= 5 and (~corrected).sum() >= 5
    for part in (corrected, ~corrected):
        assert np.abs(g[part, 8] - r[part, 8]).sum() < tol * np.abs(r[part, 8]).sum()
