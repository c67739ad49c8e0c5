"""HLLC picks the side of the contact before it forms that side's state, flux and star state (in
packed pairs for the FP32 x/y-faces): parity with the FP64 oracle on flows whose faces take all
four cases, the fan to either side of the face (supersonic both ways along every axis) and
either star state, with walls, on a uniform mesh and with a refined block, whose
faces' fluxes correct the coarse ones."""
import numpy as np
import pytest

from parity_util import TOL_FP64, force_refine, gpu_mesh, oracle_solver, rel_l1

pytestmark = pytest.mark.gpu
OUT, PER, REF = "outflow", "periodic", "reflect"
TP = 2 * np.pi


def _fast(x, y, z):
    p = np.zeros((5,) + np.shape(x))
    p[0] = 1.0 + 0.3 * np.sin(TP * (x + y + z))
    p[1] = 2.5 * np.sin(TP * y) * np.cos(TP * x)
    p[2] = 2.5 * np.sin(TP * z + 1.0) * np.cos(TP * y)
    p[3] = 2.5 * np.sin(TP * x + 2.0) * np.cos(TP * z)
    p[4] = 0.6 + 0.2 * np.cos(TP * (x - z))
    return p


@pytest.mark.parametrize("rb,tol", [(8, TOL_FP64), (4, 1e-5)])
@pytest.mark.parametrize("limiter", ["minmod", "vanleer"])
@pytest.mark.parametrize("bc", [(PER,) * 6, (OUT, OUT, REF, REF, PER, PER)])
@pytest.mark.parametrize("refine", [False, True])
def test_all_sides(rb, tol, limiter, bc, refine):
    spec = dict(physics="hd", limiter=limiter, flux="hllc", rk=2, base_blocks=(2, 2, 2), max_level=2, bc=bc)
    o = oracle_solver(spec)
    o.set_state(_fast)
    m = gpu_mesh(spec, real_bytes=rb)
    m.set_state(_fast)
    if refine:
        force_refine(o, m, {(1, 1, 0, 1)})
        m.set_state_blocks(o.get_state()[2])
    for _ in range(2):
        dt = o.cfl_dt()
        o.step(dt)
        m.step(dt)
    lev, _, g = m.get_state()
    _, _, r = o.get_state()
    m.close()
    assert set(lev) == ({1, 2} if refine else {1})
    v = r[:, 1:4] / r[:, :1]
    c = np.sqrt(5 / 9 * 2 * np.maximum(r[:, 4] - 0.5 * r[:, 0] * (v ** 2).sum(1), 0) / r[:, 0] * 1.0)
    assert np.all([(v[:, d] / c).max() > 1.2 and (v[:, d] / c).min() < -1.2 for d in range(3)])
    err = rel_l1(g, r, lev)
    assert err.max() < tol, err
