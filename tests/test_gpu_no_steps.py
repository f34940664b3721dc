"""GPU: LBMBoxFunction with no step (jets of length 0) is the initialisation and its transpose, on every handle, also one without
boundary points."""
import pytest

from paper_2410_13165_gb300 import LBM, _abi, autograd, build, jet_len

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bc", ["periodic", "fullway", "halfway"])
def test_no_steps(bc):
    import torch

    build.build()
    _abi.load()
    d, n = 2, 9
    sim = LBM(d, n, u=(0.01, 0.02), bc=bc)
    phi0 = torch.randn(n * n, dtype=torch.float64, device="cuda", requires_grad=True)
    grad = torch.randn(d * n * n, dtype=torch.float64, device="cuda", requires_grad=True)
    jets = torch.zeros(0, 1, jet_len(d), dtype=torch.float64, device="cuda", requires_grad=True)
    phi = autograd.LBMBoxFunction.apply(phi0, grad, jets, sim)
    assert (phi - phi0).abs().max() < 1e-14 * phi0.abs().max() * 9
    phi.backward(torch.ones_like(phi))
    assert (phi0.grad - 1.0).abs().max() < 1e-14 and jets.grad.shape == jets.shape
    sim.close()
