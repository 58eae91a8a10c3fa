"""The float64 reciprocal and logarithm of the sums that the float64 pipe bounds (pm_fast64.cuh)
against 64-bit-mantissa arithmetic over the exponent range, and at the special arguments.

Tolerances.  1/x: the cubic step leaves the hardware's 2^-20 to the third power and two roundings:
two ulps.  log x: the three products' roundings, each half an ulp of a term no larger than
max(|log x|, log 2), and the table's: two ulps of that."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -52


def _both(x):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2401_12501_gb300 import _lib
    x = np.ascontiguousarray(x, dtype=np.float64)
    rcp, lg = np.empty_like(x), np.empty_like(x)
    _lib.check(_lib.lib().pm_selftest_fast64(_lib.ptr(x), x.size, _lib.ptr(rcp), _lib.ptr(lg)),
               "pm_selftest_fast64")
    return rcp, lg


@pytest.mark.parametrize("lo,hi", [(-1022, 1022), (-40, 40), (-1, 1)])
def test_normal_arguments(lo, hi):
    rng = np.random.default_rng(hi)
    x = np.exp2(rng.uniform(lo, hi, 200000))
    # the ends of the table's cells and of the octaves, and their neighbours
    ends = np.ldexp(1.0 + np.arange(129) / 128.0, rng.integers(lo, hi, 129))
    x = np.concatenate([x, ends, np.nextafter(ends, 0.0), np.nextafter(ends, np.inf)])
    x = np.clip(x, 2.0 ** -1022, 2.0 ** 1021)
    rcp, lg = _both(x)
    X = x.astype(np.longdouble)
    assert (np.abs(rcp * X - 1) <= 2 * EPS).all()
    L = np.log(X)
    assert (np.abs(lg - L) <= 2 * EPS * np.maximum(np.abs(L), np.log(2.0))).all()


def test_special_arguments():
    rcp, lg = _both([0.0, np.inf, np.nan, -np.nan, 1.7e308, 2.0 ** -1030])
    assert rcp[0] == np.inf and lg[0] == -np.inf
    assert rcp[1] == 0.0 and lg[1] == np.inf
    assert np.isnan(rcp[2:4]).all() and np.isnan(lg[2:4]).all()
    assert rcp[4] == 0.0 and abs(lg[4] - np.log(1.7e308)) < 1e-12
    assert rcp[5] == np.inf and lg[5] == -np.inf
