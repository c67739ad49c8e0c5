"""The FP32 stencil's relativistic recovery finishes in FP32 pairs where their guards hold, else
in FP64. xi and Gamma of every cell of random states (read back as the auxiliaries after a step
of negligible length, which leaves the conserved state as it is) against the root found in
extended precision from the same FP32 conserved values: hot and cold gases, Lorentz factors up
to 60, both equations of state, so that cells take either branch."""
import numpy as np
import pytest

from paper_2607_19277_gb300 import agile

pytestmark = pytest.mark.gpu


def _root(cons, eos, gamma):
    """xi, Gamma from conserved values by Newton steps in extended precision from above."""
    L = np.longdouble
    D, m2, E = cons[:, 0].astype(L), (cons[:, 1:4].astype(L) ** 2).sum(1), (cons[:, 4].astype(L) + cons[:, 0])
    lo, hi = np.maximum(E, np.sqrt(m2)), (L(4) / 3 if eos == "synge" else L(gamma)) * E

    def off(x):
        w = m2 / (x * x)
        lor = 1 / np.sqrt(1 - w)
        rho = D / lor
        if eos == "synge":
            h = x / (D * lor)
            return x - rho * (5 * h - np.sqrt(9 * h * h + 16)) / 8 - E, lor
        return x - (L(gamma) - 1) / L(gamma) * (x * (1 - w) - rho) - E, lor
    for _ in range(70):                       # f rises through the root: plain bisection
        mid = (lo + hi) / 2
        up = off(mid)[0] < 0
        lo, hi = np.where(up, mid, lo), np.where(up, hi, mid)
    return hi, off(hi)[1]


@pytest.mark.parametrize("eos,gamma", [("ideal", 4.0 / 3.0), ("ideal", 5.0 / 3.0), ("synge", 4.0 / 3.0)])
@pytest.mark.parametrize("lorentz,theta", [(1.001, (-1, 1)), (10.0, (-2, 1)), (60.0, (-1, 2)), (3.0, (-4.5, -3))])
def test_recovery_against_extended_precision(eos, gamma, lorentz, theta):
    rng = np.random.RandomState(11)
    n = (2, 16, 16, 16)
    rho = 10 ** rng.uniform(-2, 2, n)
    u = rng.randn(3, *n)
    u *= np.sqrt(np.exp(rng.uniform(0, np.log(lorentz), n)) ** 2 - 1) / np.sqrt((u ** 2).sum(0))
    prim = np.stack([rho, u[0], u[1], u[2], rho * 10 ** rng.uniform(*theta, n)], axis=1)
    m = agile.Mesh(agile.make_config(physics="srhd", limiter="minmod", flux="tvdlf", rk=2, real_bytes=4, gamma=gamma,
                                     eos=eos, base_blocks=(2, 1, 1)))
    m.set_state_prims(prim)
    cons = m.get_state()[2]
    m.step(1e-35)
    assert np.array_equal(m.get_state()[2], cons)
    aux = m.get_aux()
    m.close()
    xi, lor = _root(cons, eos, gamma)
    # half an ulp of the FP32 result, and what the last step's first-order update leaves out:
    # (3/2) Gamma^4 (dxi / xi)^2 of Gamma, the step dxi being at most 1e-6 xi
    half = 2.0 ** -24 * 1.04
    assert np.all(np.abs(aux[:, 0] / xi - 1) <= half + 2e-12)
    assert np.all(np.abs(aux[:, 1] / lor - 1) <= half + 1.5 * lor ** 4 * 1e-12)


@pytest.mark.parametrize("eos,gamma", [("ideal", 4.0 / 3.0), ("ideal", 5.0 / 3.0), ("synge", 4.0 / 3.0)])
@pytest.mark.parametrize("lorentz,theta,branch", [(1.001, (-1, 1), 1), (10.0, (-2, 1), 1), (60.0, (-1, 2), 1),
                                                  (3.0, (-3.2, -2.2), 1), (3.0, (-5.5, -4.8), 0), (200.0, (0, 1), None)])
def test_density_and_pressure_against_extended_precision(eos, gamma, lorentz, theta, branch):
    """The two outputs whose cancellation the guards of the pairs are for. Bound: the FP32 rounding, 2^-29
    for the pairs, and what the last step's first-order update leaves out (as for xi and Gamma; of rho
    half of Gamma's and its own, of p through d2p/dxi2 < 4 Gamma^4 / xi). Starts a few roundings off
    the root, as a step leaves them, and far from it."""
    rng = np.random.RandomState(12)
    n = 4096
    rho = 10 ** rng.uniform(-2, 2, n)
    u = rng.randn(n, 3)
    # the upper half of the range of rapidities where the branch is to be that range's
    lor = np.exp(rng.uniform(np.log(lorentz) * (0.5 if branch is None else 0.0), np.log(lorentz), n))
    u *= (np.sqrt(lor ** 2 - 1) / np.sqrt((u ** 2).sum(1)))[:, None]
    th = 10 ** rng.uniform(*theta, n)
    g = np.sqrt(1 + (u ** 2).sum(1))
    h = 2.5 * th + np.sqrt(2.25 * th ** 2 + 1) if eos == "synge" else 1 + gamma / (gamma - 1) * th
    w = rho * h * g
    cons = np.column_stack([g * rho, w[:, None] * u, g * w - rho * th - g * rho]).astype(np.float32)
    start = np.float32(g * w) * np.float32(1 + 2.0 ** -21) * np.where(np.arange(n) % 2, np.float32(1), np.float32(1.2))
    got = agile.recover32(cons, start, gamma, eos)
    if branch is not None:
        assert (got[:, 7] == branch).mean() > 0.95, np.unique(got[:, 7], return_counts=True)
    c = cons.astype(np.float64)
    xi, lr = _root(c, eos, gamma)
    D = c[:, 0].astype(np.longdouble)
    r = D / lr
    p = xi - (c[:, 4].astype(np.longdouble) + D)
    ok = got[:, 7] >= 0
    assert ok.mean() > 0.99 and (ok.all() or branch != 1)
    ok &= p > 0
    half, out = 2.0 ** -24 * 1.04, 1e-12 * lr ** 4
    er, ep = np.abs(got[:, 0] / r - 1), np.abs(got[:, 4] / p - 1)
    assert np.all((er <= half + 2.0 ** -29 + 2 * out)[ok]), (er / (half + 2.0 ** -29 + 2 * out))[ok].max()
    assert np.all((ep <= half + 2.0 ** -29 + 2 * out * xi / p)[ok]), (ep / (half + 2.0 ** -29 + 2 * out * xi / p))[ok].max()
    if lorentz <= 10 and branch == 1:             # rms of a rounding to the nearest: 0.29 ulp
        for e, v in ((er, r), (ep, p)):
            ulp = (e * np.abs(v) / np.spacing(np.abs(v).astype(np.float32))).astype(np.float64)
            assert np.sqrt((ulp ** 2).mean()) <= 0.30


@pytest.mark.parametrize("eos,scalar", [("ideal", 4.106e-7), ("synge", 8.375e-7)])
def test_energy_of_a_cold_gas(eos, scalar):
    """tau = Gamma^2 rho h - p - D cancels in a cold gas: FP32 against FP64 steps from the same state. The
    FP32 pairs of the face solver leave tau no further off than 1.04 times what the scalar FP32 solver,
    in which the compiler fuses the products into the sums, was measured to leave."""
    t = 2 * np.pi

    def ic(x, y, z):
        p = np.zeros((5,) + np.shape(x))
        p[0] = 1.0 + 0.3 * np.sin(t * (x + 2 * y - z))
        p[1], p[2], p[3] = 0.05 * np.sin(t * y + 0.3), 0.05 * np.cos(t * z), 0.05 * np.sin(t * x + 1)
        p[4] = 1e-3 * (1.0 + 0.3 * np.cos(t * (x - z)))
        return p

    out = {}
    for rb in (4, 8):
        m = agile.Mesh(agile.make_config(physics="srhd", limiter="vanleer", flux="tvdlf", rk=2, real_bytes=rb,
                                         gamma=4.0 / 3.0, eos=eos, base_blocks=(3, 3, 3)))
        m.set_state(ic)
        if rb == 4:
            start = m.get_state()[2]
        else:
            m.set_state_blocks(start)
        for _ in range(6):
            m.step(2e-3)
        out[rb] = m.get_state()[2][:, 4]
        m.close()
    err = np.sqrt(((out[4] - out[8]) ** 2).mean() / (out[8] ** 2).mean())
    assert err <= 1.04 * scalar, err
