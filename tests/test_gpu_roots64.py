"""The FP64 stencil's roots, refined from the hardware estimate, against extended precision: the root
of one argument and of a quotient, over the exponents the stencil meets and beyond, mantissas next
to powers of two, and on both sides of the limits outside which other forms are taken. The bounds
are those of the interface: half an ulp for the last addition, 0.02 for the terms of the series
left out; for a quotient w = b s is rounded as well, 2^-54 of the result, at most half an ulp; by the
other form the reciprocal and the product are (2^-53 of the result, at most one ulp). A correctly
rounded result has rms 1 / sqrt(12) ulp."""
import numpy as np
import pytest

from paper_2607_19277_gb300 import agile

pytestmark = pytest.mark.gpu
N = 1 << 18
L = np.longdouble


def _values(rng, lo, hi):
    a = np.ldexp(1.0 + rng.random(N), rng.integers(lo, hi, N))
    near = np.ldexp(1.0, rng.integers(lo, hi, N // 8)) * (1.0 + 2.0 ** -52 * rng.integers(-4, 8, N // 8))
    return np.concatenate([a, near])


def _ulps(got, ref):
    return np.abs((got.astype(L) - ref) / np.spacing(ref.astype(np.float64)).astype(L)).astype(np.float64)


@pytest.mark.parametrize("lo,hi", [(-4, 4), (-300, 300), (-1022, 1023), (-965, -953)])
def test_root(lo, hi):
    a = _values(np.random.default_rng(3), lo, hi)
    u = _ulps(agile.eval_fp64("sqrt", a), np.sqrt(a.astype(L)))
    assert u.max() <= 0.52, u.max()
    assert np.sqrt((u ** 2).mean()) <= 0.2905


def test_root_of_squares_and_special_values():
    n = np.concatenate([np.arange(1.0, 3000.0), np.ldexp(1.0, np.arange(-480, 500)), [3.0 * 2.0 ** 25 + 1.0]])
    assert np.array_equal(agile.eval_fp64("sqrt", n * n), n)
    tiny = np.finfo(np.float64).tiny
    a = np.array([0.0, -0.0, 5e-324, tiny / 2, tiny, 2.0 ** -960, 2.0 ** -959, np.finfo(np.float64).max, np.inf])
    got = agile.eval_fp64("sqrt", a)
    assert np.array_equal(got, np.sqrt(a)) and np.signbit(got[1])
    assert np.all(np.isnan(agile.eval_fp64("sqrt", np.array([-1.0, -5e-324, -np.inf, np.nan]))))


@pytest.mark.parametrize("lo,hi", [(-4, 4), (-300, 300), (-450, 450)])
def test_root_of_a_quotient(lo, hi):
    rng = np.random.default_rng(4)
    a, b = _values(rng, lo, hi), _values(rng, lo, hi)
    u = _ulps(agile.eval_fp64("sqrt_quotient", a, b), np.sqrt(a.astype(L) / b.astype(L)))
    assert u.max() <= 1.02, u.max()
    # no larger than by the rounded quotient's correctly rounded root: rms of (1, 1, 2) / 2 roundings
    assert np.sqrt((u ** 2).mean()) <= 0.36


@pytest.mark.parametrize("ea,eb", [(-512, -512), (-600, -520), (510, 510), (700, 700), (-960, 0), (-1000, -400), (-959, 50)])   # a / b normal everywhere
def test_root_of_a_quotient_at_the_limits(ea, eb):
    rng = np.random.default_rng(5)
    a, b = _values(rng, ea - 3, ea + 4), _values(rng, eb - 3, eb + 4)
    u = _ulps(agile.eval_fp64("sqrt_quotient", a, b), np.sqrt(a.astype(L) / b.astype(L)))
    assert u.max() <= 1.55, u.max()


def test_root_of_a_quotient_special_values():
    got = agile.eval_fp64("sqrt_quotient", np.array([0.0, 5e-324, np.inf]), np.array([3.0, 2.0 ** -1000, 2.0]))
    assert got[0] == 0.0 and got[1] == pytest.approx(np.sqrt(5e-324 * 2.0 ** 1000), rel=1e-15) and got[2] == np.inf
    assert np.all(np.isnan(agile.eval_fp64("sqrt_quotient", np.array([-1.0, 1.0, -5e-324, np.nan]),
                                           np.array([1.0, -1.0, 1.0, 1.0]))))
