"""A mesh that does not fit the device is refused for want of memory."""
import pytest

from paper_2508_13705_gb300 import cgks


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
