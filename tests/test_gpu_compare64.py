"""The FP64 stencil's minima, maxima and sign tests run on the bit patterns: the same results as the
floating-point comparisons for every pair of numbers, infinities, subnormals and signed zeros
included; of a NaN and a number the number."""
import numpy as np
import pytest

from paper_2607_19277_gb300 import agile

pytestmark = pytest.mark.gpu


def _values():
    rng = np.random.default_rng(6)
    tiny, big = np.finfo(np.float64).tiny, np.finfo(np.float64).max
    nans = np.array([0x7ff8000000000000, 0xfff8000000000000, 0x7ff0000000000001, 0xffffffffffffffff],
                    dtype=np.uint64).view(np.float64)
    one = [0.0, 5e-324, tiny / 2, tiny, 1.0, 1.0 + 2.0 ** -52, 2.0, 1e300, big, np.inf]
    return np.concatenate([one, np.negative(one), nans, rng.normal(0, 1, 40), rng.integers(0, 2 ** 63, 60).astype(np.uint64).view(np.float64)])


def _same(got, want):
    nan = np.isnan(want)
    assert np.array_equal(np.isnan(got), nan)
    assert np.array_equal(got[~nan].view(np.uint64), want[~nan].view(np.uint64))


def test_minimum_and_maximum():
    v = _values()
    a, b = (x.ravel() for x in np.meshgrid(v, v))
    with np.errstate(invalid="ignore"):
        lo = np.where(np.isnan(a), b, np.where(np.isnan(b) | (a < b), a, b))
        hi = np.where(np.isnan(a), b, np.where(np.isnan(b) | (a > b), a, b))
    zeros = (a == 0) & (b == 0)                   # of two zeros -0 is the smaller
    lo[zeros] = np.where(np.signbit(a[zeros]) | np.signbit(b[zeros]), -0.0, 0.0)
    hi[zeros] = np.where(np.signbit(a[zeros]) & np.signbit(b[zeros]), -0.0, 0.0)
    _same(agile.eval_fp64("min", a, b), lo)
    _same(agile.eval_fp64("max", a, b), hi)


def test_sign_tests():
    v = _values()
    with np.errstate(invalid="ignore"):
        assert np.array_equal(agile.eval_fp64("positive", v) == 1, v > 0)
        assert np.array_equal(agile.eval_fp64("not_nonnegative", v) == 1, ~(v >= 0))
