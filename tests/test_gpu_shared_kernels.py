"""Solvers of one process share their kernels: what one solver sets on a kernel
must leave the launches of the others as they are."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2508_13705_gb300 import cgks, inputs  # noqa: E402


def test_tuned_solvers_of_one_kernel_keep_stepping():
    """Autotuned solvers whose tile shapes may differ, in bytes of shared
    memory too: each still steps after all are tuned, with equal results."""
    n = 96
    st = inputs.vortex_2d(n, 9)
    solvers = []
    for k in range(12):
        s = cgks.Solver(2, 9, n, n, extent=(0, 10, 0, 10), precision=cgks.FP32_BULK)
        s.set_state(*st)
        if k:  # the first keeps the default tile, one of the largest
            s.autotune()
        solvers.append(s)
    dt = solvers[0].compute_dt()
    want = None
    for s in solvers:
        s.step(dt)
        s.sync()
        W = s.get_state()["W"]
        want = W if want is None else want
        assert np.array_equal(W, want)
        s.close()
