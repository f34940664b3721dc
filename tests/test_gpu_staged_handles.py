"""GPU: staged handles of several grids at once. Their kernels' shared-memory limit belongs to the process: a handle created later,
with smaller stages, must not take it away from an earlier one."""
import pytest

from paper_2410_13165_gb300 import LBM, _abi, build

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("adjoint", [False, True])
def test_a_later_handle_leaves_the_earlier_one_running(adjoint):
    import torch

    build.build()
    _abi.load()
    n = (256, 128, 128)
    x = torch.sin(torch.arange(256 * 128 * 128, dtype=torch.float64, device="cuda") * 0.01)
    out = []
    for later in (None, (128, 128, 112)):
        a = LBM(3, list(n), 0.0, [m / 128.0 for m in n], u=(0.1, 0.1, 0.1), precision="fp32dev")
        b = None if later is None else LBM(3, list(later), 0.0, [m / 128.0 for m in later], u=(0.1, 0.1, 0.1), precision="fp32dev")
        a.init(x)
        a.step(2)
        if adjoint:
            a.adjoint_seed(x)
            a.adjoint_step(2)
        out.append(a.get_state().clone())
        a.close()
        if b is not None:
            b.close()
    assert torch.equal(*out)
