"""The FP64 hydro speed sqrt(gamma p / rho) takes the root of the product p rho where that is a
normal number and the quotient's root elsewhere: a state scaled by a power of two (density,
momentum and energy; the equations are homogeneous in it) that takes p rho out of that range
gives the scaled results. Each of the two roots is within 2 ulp, and the stencil damps a speed's error to its
share of the flux, so two steps stay within 1e-14 of one another."""
import numpy as np
import pytest

from paper_2607_19277_gb300 import agile, workloads as W

pytestmark = pytest.mark.gpu


def _steps(scale, flux):
    m = agile.Mesh(agile.make_config(physics="hd", limiter="minmod", flux=flux, rk=2, real_bytes=8,
                                     base_blocks=(2, 2, 2)))
    ic = W.random_smooth(5, 11, "hd")

    def scaled(x, y, z):
        p = np.array(ic(x, y, z))
        p[[0, 4]] *= scale
        return p

    m.set_state(scaled)
    for _ in range(2):
        m.step()
    cons = m.get_state()[2]
    m.close()
    return cons


@pytest.mark.parametrize("flux", ["tvdlf", "hll"])
@pytest.mark.parametrize("exponent", [-600, -511, 500, 600])
def test_scaled_state(flux, exponent):
    one = _steps(1.0, flux)
    got = _steps(2.0 ** exponent, flux) * 2.0 ** -exponent
    for v in range(5):
        err = np.abs(got[:, v] - one[:, v]).sum() / max(np.abs(one[:, v]).sum(), np.abs(one[:, 0]).sum())
        assert err < 1e-14, (v, err)
