"""The square root and the reciprocals of the Cholesky kernels (their own short
chains in place of sqrt and a division) against IEEE 754 square root and division,
bit for bit: random mantissas at every exponent, mantissas of all ones, all zeros
and their neighbours, the exponents at which the long way takes over, the ends of
the range, and what has no root."""
import numpy as np
import pytest

import paper_2607_15158_gb300 as pkg

pytestmark = pytest.mark.gpu


def _check(x):
    root, rroot, rcp = pkg.ctm_debug_roots(x)
    with np.errstate(all="ignore"):
        r = np.sqrt(x)
        want = (r, 1.0 / r, 1.0 / x)
    for got, w in zip((root, rroot, rcp), want):
        nan = np.isnan(w)
        assert np.array_equal(np.isnan(got), nan)
        assert np.array_equal(got[~nan].view(np.int64), w[~nan].view(np.int64))


def _value(field, mantissa):
    return ((np.asarray(field, np.uint64) << np.uint64(52)) | np.asarray(mantissa, np.uint64)).view(
        np.float64)


@pytest.mark.parametrize("seed", range(4))
def test_random_mantissas_at_every_exponent(seed):
    rng = np.random.default_rng(seed)
    n = 1 << 21
    _check(_value(rng.integers(0, 2047, n), rng.integers(0, 1 << 52, n)))
    # the range of the pivots and the column scales
    _check(_value(rng.integers(1023 - 60, 1023 + 60, n), rng.integers(0, 1 << 52, n)))


def test_special_mantissas_at_every_exponent():
    top = 1 << 52
    m = [0, 1, 2, 3, top - 1, top - 2, top - 3, top // 2, top // 2 - 1, top // 2 + 1]
    m += [(1 << i) for i in range(52)] + [top - (1 << i) for i in range(52)]
    f, mm = np.meshgrid(np.arange(2047), np.array(m, np.uint64), indexing="ij")
    x = _value(f.ravel(), mm.ravel())
    _check(x)
    # roots of all ones: squares of values just below a power of two, and neighbours
    r = _value(np.arange(512, 1535), np.full(1023, top - 1))
    s = r * r
    for step in range(-3, 4):
        _check((s.view(np.int64) + step).view(np.float64))


def test_what_has_no_root():
    _check(np.array([0.0, -0.0, np.inf, -np.inf, np.nan, -1.0, 5e-324, -5e-324, -1e300, 2.2e-308]))
