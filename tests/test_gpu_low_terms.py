"""GPU: FP64 moment sums of very small terms and of zeros: a field scaled down by a power of two steps to the scaled result
(1D: bit for bit), and regions of zeros are stepped no slower than others."""
import numpy as np
import pytest

from paper_2410_13165_gb300 import LBM, _abi, build

pytestmark = pytest.mark.gpu
U = (0.05, 0.04, 0.03, 0.02, 0.01)


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    _abi.load()


def _state(d, n, tau, bc, x, steps, adjoint):
    import torch

    hi = [m - 1.0 if bc == "fullway" else float(m) for m in n]
    sim = LBM(d, n, hi=hi, u=U[:d], tau=tau, bc=bc)
    if bc == "periodic":
        sim.init(x)
    else:
        sim.init(x, torch.zeros(d * x.numel(), dtype=torch.float64, device="cuda"))
        sim.set_boundary_wave()
    sim.step(steps)
    out = [sim.get_state().clone().view(torch.float64), sim.macro()]
    if adjoint:
        sim.adjoint_seed(x)
        sim.adjoint_step(steps)
        out.append(sim.adjoint_grads(want_R=True)[2])
    sim.close()
    return out


# 2^-960: every term below 2^-954 from the start; 2^-950: on either side of it
@pytest.mark.parametrize("shift", [950, 960])
@pytest.mark.parametrize("tau", [0.5, 0.8])
@pytest.mark.parametrize("d,n,bc", [(1, (70,), "periodic"), (2, (12, 9), "periodic"), (2, (300, 230), "periodic"), (3, (9, 10, 7), "periodic"),
                                    (4, (6, 5, 4, 7), "periodic"), (5, (5, 4, 3, 4, 5), "periodic"), (3, (9, 8, 7), "fullway"),
                                    (4, (5, 6, 5, 4), "halfway")])
def test_small_fields_step_like_scaled_ones(d, n, bc, tau, shift):
    import torch

    rng = np.random.default_rng(d)
    # (values within a factor 2^10 of one another, so that scaled terms keep all their bits: the smallest stay above 2^-1000)
    x = torch.from_numpy(rng.uniform(0.5, 2.0, int(np.prod(n))) * rng.choice([1.0, 2.0 ** -8], int(np.prod(n)))).cuda()
    small = 2.0 ** -shift
    a = _state(d, n, tau, bc, x, 3, bc == "periodic")
    b = _state(d, n, tau, bc, x * small, 3, bc == "periodic")
    Q = 2 * d * d + 1
    for p, q in zip(a, b):
        if d == 1:
            assert torch.equal(p * small, q)
        else:  # a sum of Q terms in FP64 is within Q / 2 units of the largest; three steps each way, on sums of at most Q x 2
            assert (p * small - q).abs().max() <= 6 * Q * Q * 2.0 ** -53 * small


@pytest.mark.parametrize("d,n,bc", [(2, 1000, "periodic"), (3, 128, "periodic"), (4, 32, "periodic"), (5, 16, "periodic"), (3, 100, "fullway"),
                                    (4, 24, "halfway")])
def test_zeros_are_stepped_no_slower(d, n, bc):
    import torch

    ms = []
    for zero in (False, True):
        sim = LBM(d, n, hi=float(n - 1 if bc == "fullway" else n), u=U[:d], tau=0.8, bc=bc)
        x = torch.ones(n ** d, dtype=torch.float64, device="cuda") * (0.0 if zero else 1.0)
        if bc == "periodic":
            sim.init(x)
        else:
            sim.init(x, torch.zeros(d * n ** d, dtype=torch.float64, device="cuda"))
            sim.set_boundary_wave(b=0.0 if zero else 1.0)
        sim.step(8)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        best = 1e30
        for _ in range(7):
            e0.record()
            sim.step(16)
            e1.record()
            e1.synchronize()
            best = min(best, e0.elapsed_time(e1))
        ms.append(best)
        sim.close()
    assert ms[1] < 1.15 * ms[0], ms
