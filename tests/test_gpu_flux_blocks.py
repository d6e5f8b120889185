"""Solvers of one kernel set whose flux launches differ in block size, and with it
in dynamic shared memory (a kernel's limit on it belongs to the kernel, not to the
solver): a tiny mesh with a warp a block, a larger one with four, and tuned ones,
made, tuned and stepped in turn."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2508_13705_gb300 import cgks, inputs  # noqa: E402


@pytest.mark.parametrize("tau", [cgks.TAU_ZERO, cgks.TAU_HGKS])
@pytest.mark.parametrize("order,precision", [(5, cgks.FP32_BULK), (7, cgks.FP64), (9, cgks.FP32_BULK), (9, cgks.FP64)])
def test_solvers_with_other_block_sizes_keep_stepping(order, precision, tau):
    sizes = (8, 96)
    states = {n: inputs.vortex_2d(n, order) for n in sizes}
    kw = dict(extent=(0, 10, 0, 10), precision=precision, tau_mode=tau)

    def step(s, dt):
        s.step(dt)
        s.sync()
        return s.get_state()["W"]

    dt, want = {}, {}
    for n in sizes:  # each mesh alone, untuned
        s = cgks.Solver(2, order, n, n, **kw)
        s.set_state(*states[n])
        dt[n] = s.compute_dt()
        want[n] = [step(s, dt[n]) for _ in range(2)]
        s.close()
    solvers = []
    for k in range(6):
        n = sizes[k % 2]
        s = cgks.Solver(2, order, n, n, **kw)
        s.set_state(*states[n])
        if k >= 2:
            s.autotune()
        solvers.append((n, s))
        for m, t in solvers[:1] + solvers[-1:]:  # the first keeps up with the last
            t.set_state(*states[m])
            assert np.array_equal(step(t, dt[m]), want[m][0])
    for n, s in solvers:
        s.set_state(*states[n])
    for i in range(2):
        for n, s in reversed(solvers):
            assert np.array_equal(step(s, dt[n]), want[n][i])
    for _, s in solvers:
        s.close()
