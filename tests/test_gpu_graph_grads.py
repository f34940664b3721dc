"""GPU: lhe_lbm_adjoint_grads allocates nothing after lhe_lbm_adjoint_seed, also when the library formed the gradient of phi0
itself, so that it can be captured into a graph."""
import pytest

from paper_2410_13165_gb300 import LBM, _abi, build

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32dev"])
def test_gradients_in_a_graph(precision):
    import torch

    build.build()
    _abi.load()
    sim = LBM(3, 16, u=(0.1, 0.1, 0.1), precision=precision)
    g = torch.Generator(device="cuda").manual_seed(1)
    x, seed = (torch.randn(16 ** 3, dtype=torch.float64, device="cuda", generator=g) for _ in range(2))

    def adjoint():
        sim.init(x)
        sim.step(3)
        sim.adjoint_seed(seed)
        sim.adjoint_step(3)

    adjoint()
    out = torch.zeros(16 ** 3, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        sim._stream()
        _abi.lhe_lbm_adjoint_grads(sim.h, out.data_ptr(), None, None)
    graph.replay()
    torch.cuda.synchronize()
    adjoint()
    want = sim.adjoint_grads(want_R=False)[0]
    assert torch.equal(out, want)
    sim.close()
