"""FP32 bulk: the stage-1 averages W* are formed by one FP64 subtraction from the
FP64 averages and only then split into hi + lo.

The flux sums are floats, the spacing is a power of two and the y fluxes are
equal, so that what is subtracted is exact and W* is one rounding in FP64:
compared bit for bit."""
import ctypes

import numpy as np
import pytest

import kernel_units

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("size", [1e-7, 1e-3, 1.0])
@pytest.mark.parametrize("nx,ny", [(1, 1), (37, 9), (256, 3)])
def test_star_averages_are_fp64_differences(nx, ny, size):
    rng = np.random.default_rng(nx + ny)
    h = 2.0**-4
    # one base for all cells (no flux differences of the bases), FP64 tails of their own
    base = np.array([1.0, 0.7, -0.3, 2.5])[:, None, None]
    W = base.astype(np.float32).astype(np.float64) * (1 + 2.0**-26 * rng.uniform(-1, 1, (4, ny, nx)))
    f = (size * rng.uniform(-1, 1, (ny, nx + 1, 4))).astype(np.float32)
    hi, lo = np.empty((2, 4, ny, nx), np.float32)
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)
    assert kernel_units.lib().unit_stage1_averages(nx, ny, ctypes.c_double(h), p(W), p(f), p(hi), p(lo)) == 0
    d = (f[:, 1:].astype(np.float64) - f[:, :-1]) / h
    want = W - np.moveaxis(d, -1, 0)
    whi = want.astype(np.float32)
    assert np.array_equal(hi, whi)
    assert np.array_equal(lo, (want - whi).astype(np.float32))
