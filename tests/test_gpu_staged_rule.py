"""GPU: which FP32-deviation kernel a periodic D3Q19 grid takes must not show: on either side of the lines of the rule
(forward and adjoint chosen apart), the default handle and the register kernel give the same bits."""
import numpy as np
import pytest

from paper_2410_13165_gb300 import LBM, _abi, build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    _abi.load()


@pytest.mark.parametrize("n", [(128, 112, 128), (128, 108, 128), (256, 64, 64), (256, 62, 64), (64, 128, 128), (100, 100, 105), (96, 100, 112)])
@pytest.mark.parametrize("tau", [0.5, 0.8])
def test_default_kernels_are_bitwise_the_register_kernel(n, tau):
    import torch

    rng = np.random.default_rng(sum(n))
    phi0, R, seed = (torch.from_numpy(rng.standard_normal(int(np.prod(n)))).cuda() for _ in range(3))
    out = []
    for staged in (True, False):
        sim = LBM(3, list(n), 0.0, [m / 64.0 for m in n], u=(0.1, -0.05, 0.08), tau=tau, precision="fp32dev", staged=staged)
        sim.init(phi0, None, R)
        sim.step(3)
        got = [sim.get_state().clone()]
        sim.adjoint_seed(seed)
        sim.adjoint_step(3)
        gphi, _, gR = sim.adjoint_grads(want_grad=False, want_R=True)
        out.append(got + [gphi, gR])
        sim.close()
    for a, b in zip(*out):
        assert torch.equal(a, b)
