"""The 2-D flux kernel marches warps over strips of 32 / m faces (16, 10, 8 for
orders 5, 7, 9), and Steps 1-2 cover the mesh and a ring of ghost cells with
tiles of 28 x 4 (x faces; FP64 28 x 2) and 12 x 16 (y faces; FP64 12 x 8) cells: meshes that
fill strips or tiles exactly, fall one short or spill one over, in each
direction, alone and as a batch (one work list over meshes of different sizes),
against the oracle after one step.

Tolerances: FP64 1e-12 relative L1 with every value within 1e-11 of the field's
largest (the operation order differs); FP32 bulk 2e-7 for the averages and 1e-4
for slopes, the stated per-step bounds of that form."""
import numpy as np
import pytest

import oracle
from paper_2508_13705_gb300 import cgks, inputs

pytestmark = pytest.mark.gpu
FIELDS = ("W", "Wx", "Wy", "Wx_line", "Wy_line")


def wave(nx, ny, order):
    ext = (0.0, 2.0, 0.0, 2.0 * ny / nx)

    def prim(x, y):
        s = np.sin(np.pi * x) * np.cos(2 * np.pi * y / ext[3])
        return 1 + 0.2 * s, 1 + 0.1 * s, 0.7 - 0.1 * s, 1 + 0.05 * s
    return inputs.cell_state_2d(prim, nx, ny, ext, order), ext


def check(got, orc, precision, what):
    ref = orc.get_state()
    h = min(orc.dx, orc.dy)
    for f in FIELDS:
        d, r = np.abs(got[f] - ref[f]), np.abs(ref[f])
        tol = 1e-12 if precision == cgks.FP64 else (2e-7 if f == "W" else 1e-4)
        # the oracle forms slopes by a fit that leaves ulps of the state in them
        floor = 0.0 if f == "W" else 64 * np.finfo(float).eps * np.abs(ref["W"]).max() / h
        assert d.sum() <= tol * r.sum() + d.size * floor, (what, f, d.sum() / r.sum())
        assert d.max() <= 10 * tol * r.max() + floor, (what, f, d.max() / r.max())


def sizes(order):
    fw = 32 // {5: 2, 7: 3, 9: 4}[order]
    return [(fw - 2, fw + 1), (fw - 1, fw), (fw, fw - 1), (fw + 1, 2 * fw), (2 * fw - 1, 3), (3, 2 * fw + 1),
            (26, 14), (27, 10), (25, 22), (54, 6)]


@pytest.mark.parametrize("precision", [cgks.FP64, cgks.FP32_BULK])
@pytest.mark.parametrize("tau,bc", [(cgks.TAU_ZERO, (0, 0, 0, 0)), (cgks.TAU_HGKS, (1, 3, 4, 1))])
@pytest.mark.parametrize("order", [5, 7, 9])
def test_strip_edges(order, tau, bc, precision):
    oracle.build()
    dims = sizes(order)
    states = [wave(nx, ny, order) for nx, ny in dims]
    batch = cgks.Batch(order, [d[0] for d in dims], [d[1] for d in dims], [e for _, e in states], precision=precision,
                       tau_mode=tau, bc=bc)
    dts = []
    for k, ((nx, ny), (st, ext)) in enumerate(zip(dims, states)):
        batch.set_state(k, *st)
        o = oracle.Oracle(2, order, nx, ny, extent=ext, tau_mode=tau, bc=bc)
        o.set_state(*st)
        dt = o.compute_dt()
        dts.append(dt)
        o.step(dt)
        s = cgks.Solver(2, order, nx, ny, extent=ext, precision=precision, tau_mode=tau, bc=bc)
        s.set_state(*st)
        s.step(dt)
        s.sync()
        check(s.get_state(), o, precision, (nx, ny))
        s.close()
        states[k] = o
    batch.step(dts)
    batch.sync()
    for k, o in enumerate(states):
        check(batch.get_state(k), o, precision, ("batch",) + dims[k])
    batch.close()
