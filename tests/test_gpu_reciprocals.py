"""The FP32 reciprocal and reciprocal square root of the flux kernels against 64
bits, over the exponents for which argument and result are normal numbers.

Bounds, from the stated errors of the approximations (rcp.approx 1 ulp, rsqrtf 2
ulp) and one Newton-Raphson step each: recip squares its relative error of at
most 2^-23 and rounds the residual to 2^-24 of it, less than 2^-45 before the last
rounding, so 0.5 + 2^-21 ulp.  recip_sqrt adds half the rounding of x r, 2^-25
relative, which is m / 4 ulp for a result of mantissa m in [1, 2), to terms below
2^-42: 0.5 + m / 4 + 2^-18 ulp."""
import ctypes

import numpy as np
import pytest

import kernel_units

pytestmark = pytest.mark.gpu


def values(x):
    x = np.ascontiguousarray(x, np.float32)
    r, q = np.empty_like(x), np.empty_like(x)
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)
    assert kernel_units.lib().unit_reciprocals(p(x), p(r), p(q), x.size) == 0
    return x.astype(np.float64), r, q


def ulps(got, ref):
    """Error in units of the reference's last place, and its mantissa in [1, 2)."""
    m, e = np.frexp(np.abs(ref))
    return np.abs(got.astype(np.float64) - ref) / np.ldexp(1.0, e - 24), 2 * m


def arguments():
    rng = np.random.default_rng(7)
    mantissa = np.concatenate([1 + rng.random(4000), 1 + np.arange(8) * 2.0**-23, 2 - np.arange(1, 9) * 2.0**-23])
    return (mantissa[None, :] * 2.0 ** np.arange(-125, 126)[:, None]).ravel()


def test_reciprocal():
    x = arguments()
    x, r, _ = values(np.concatenate([x, -x]))
    err, _ = ulps(r, 1.0 / x)
    assert err.max() <= 0.5 + 2.0**-21, (err.max(), x[err.argmax()])
    assert np.all(np.sign(r) == np.sign(x))


def test_reciprocal_square_root():
    x, _, q = values(arguments())
    err, m = ulps(q, 1.0 / np.sqrt(x))
    assert np.all(err <= 0.5 + m / 4 + 2.0**-18), (err.max(), x[(err - m / 4).argmax()])


def test_no_reciprocal_of_zero_or_infinity():
    _, r, _ = values([0.0, -0.0, np.inf, -np.inf, np.nan])
    assert np.all(np.isnan(r))
