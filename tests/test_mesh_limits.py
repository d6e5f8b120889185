"""Meshes at the limit of the sizes that are taken (1-D: 2^31 - 3 cells): the
scratch rows are counted in 64 bits, and a mesh that does not fit the device is
refused for want of memory."""
import pytest

import kernel_units
from paper_2508_13705_gb300 import cgks

SIZES = [2**31 - 9, 2**31 - 8, 2**31 - 4, 2**31 - 3]


@pytest.mark.parametrize("nx", SIZES)
def test_face_state_rows_of_the_longest_meshes(nx):
    """Three rows of nx + 1 faces, padded to 8."""
    assert kernel_units.lib().unit_fr_nrow(0, nx, 1) == 3 * ((nx + 1 + 7) // 8 * 8)


@pytest.mark.gpu
@pytest.mark.parametrize("precision", [cgks.FP64, cgks.FP32_BULK])
@pytest.mark.parametrize("nx", SIZES)
def test_longest_meshes_are_refused_for_memory(nx, precision):
    """584 bytes a cell and more: over 1 TB."""
    with pytest.raises(cgks.CgksError) as e:
        cgks.Solver(1, 5, nx, precision=precision)
    assert e.value.code == cgks.ENOMEM


@pytest.mark.gpu
def test_refused_mesh_leaves_no_error_behind():
    """The refusal is the call's result alone: the process's other CUDA code
    does not meet it again."""
    torch = pytest.importorskip("torch")
    x = torch.zeros(1000, device="cuda")
    with pytest.raises(cgks.CgksError) as e:
        cgks.Solver(1, 5, 2**31 - 9)
    assert e.value.code == cgks.ENOMEM
    assert float((x + 1).sum()) == 1000.0
