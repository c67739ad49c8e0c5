"""The FP64 signal speeds are formed from products that have the square of the state's scale: the
hydro speed sqrt(gamma p / rho) from the root of p rho where that is a normal number and from the
quotient's root elsewhere, the MHD face's fast speed from S = gamma p + B^2 where S^2 keeps its
bits and from quantities divided by the density elsewhere. The equations are homogeneous: a state
scaled by a power of two (density, momentum and energy by s, B and psi by sqrt(s)) gives the scaled
results, also where it takes those products out of the range. Each of the roots is within 2 ulp,
and the stencil damps a speed's error to its share of the flux, so two steps stay within 1e-14 of
one another."""
import numpy as np
import pytest

from paper_2607_19277_gb300 import agile, workloads as W

pytestmark = pytest.mark.gpu


def _steps(physics, exponent, flux):
    nv = agile.NVAR[agile.PHYSICS[physics]]
    by = np.ldexp(1.0, np.where(np.arange(nv) >= 5, exponent // 2, np.where(np.arange(nv) % 4, 0, exponent)))
    m = agile.Mesh(agile.make_config(physics=physics, limiter="minmod", flux=flux, rk=2, real_bytes=8,
                                     base_blocks=(2, 2, 2)))
    ic = W.random_smooth(nv, 11, physics)
    m.set_state(lambda x, y, z: (np.array(ic(x, y, z)).T * by).T)   # rho, p by s; B, psi by sqrt(s)
    for _ in range(2):
        m.step()
    cons = m.get_state()[2]
    m.close()
    return cons


@pytest.mark.parametrize("flux", ["tvdlf", "hll"])
@pytest.mark.parametrize("physics,exponent", [("hd", -600), ("hd", -511), ("hd", 500), ("hd", 600),
                                              ("mhd", -600), ("mhd", -510), ("mhd", -400), ("mhd", 500), ("mhd", 600)])
def test_scaled_state(physics, flux, exponent):
    one = _steps(physics, 0, flux)
    got = _steps(physics, exponent, flux)
    for v in range(one.shape[1]):
        back = np.ldexp(got[:, v], -(exponent // 2 if v >= 5 else exponent))
        own = np.abs(one[:, v]).sum()
        err = np.abs(back - one[:, v]).sum() / max(own, np.abs(one[:, 5 if v >= 5 else 0]).sum())
        assert err < 1e-14, (v, err)
