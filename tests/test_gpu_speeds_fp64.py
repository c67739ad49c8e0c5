"""Signal speeds of the FP64 stencil (square roots refined from the hardware estimate, maxima on
bit patterns) from uniform states of widely spread size: one block per state, the CFL step of
every solve of a batch against the formula. The sound speed carries the rounding of gamma p, the
quotient (1 ulp) and the root (1 ulp), the sum and the quotients by dx a few more."""
import numpy as np
import pytest

from paper_2607_19277_gb300 import agile, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("physics", ["hd", "mhd"])
def test_cfl_of_uniform_states(physics):
    rng = np.random.RandomState(3)
    n, nv = 120, agile.NVAR[agile.PHYSICS[physics]]
    scale = 10.0 ** rng.uniform(-60, 60, n)           # p and rho far from one, p / rho too
    p = np.zeros((n, nv))
    p[:, 0] = 10.0 ** rng.uniform(-60, 60, n)
    p[:, 4] = p[:, 0] * scale
    p[:, 1:4] = rng.randn(n, 3) * np.sqrt(scale)[:, None] * 10.0 ** rng.uniform(-3, 1, (n, 1))
    if physics == "mhd":
        p[:, 5:8] = rng.randn(n, 3) * np.sqrt(p[:, 4])[:, None] * 10.0 ** rng.uniform(-3, 1, (n, 1))
        p[0, 5:8] = 0.0                               # the inner root of the fast speed is exact
        p[1, 6:8] = 0.0
        p[1, 5] = np.sqrt(5.0 / 3.0 * p[1, 4])        # ... and its argument cancels to zero here
    cfg = agile.make_config(physics=physics, limiter="minmod", flux="hll", rk=2, real_bytes=8, base_blocks=(1, 1, 1))
    b = agile.Batch([cfg] * n)
    for i in range(n):
        b.set_state(i, W.uniform_state(p[i]))
    dt = b.cfl_dt()
    b.close()
    L = np.longdouble
    q = p.astype(L)
    a2 = L(cfg.gamma) * q[:, 4] / q[:, 0]
    tot = L(0)
    for d in range(3):
        c2 = a2
        if physics == "mhd":
            s = a2 + (q[:, 5:8] ** 2).sum(1) / q[:, 0]
            c2 = (s + np.sqrt(np.maximum(s * s - 4 * a2 * q[:, 5 + d] ** 2 / q[:, 0], 0))) / 2
        tot = tot + (np.abs(q[:, 1 + d]) + np.sqrt(c2)) * 16
    want = L(cfg.cfl) / tot
    # the pressure is recovered from the energy, whose rounding the kinetic and magnetic parts
    # amplify; a cancelled root's argument is sqrt(ulp)-accurate
    amp = 1 + (0.5 * p[:, 0] * (p[:, 1:4] ** 2).sum(1) + (0.5 * (p[:, 5:8] ** 2).sum(1) if physics == "mhd" else 0)) / p[:, 4]
    tol = 2.0 ** -53 * (12 + 8 * amp)
    if physics == "mhd":
        tol[1] = 2.0 ** -24
    assert np.all(np.abs(dt / want - 1) <= tol), np.max(np.abs(dt / want - 1) / tol)
