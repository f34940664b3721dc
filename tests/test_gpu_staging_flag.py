"""GPU: LHE_FLAG_STAGING runs the staged FP32-deviation step on every grid its layout admits, so that it is compared with the
register kernel (single steps without staging) and the several-steps kernel (calls of many steps) where neither rule would choose
it: tiles of one and several rows, rows that do not divide a unit of 32 nodes, wrap-around on 3 rows, 512 nodes a row."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2410_13165_gb300 import LBM, LHEError, _abi, build

pytestmark = pytest.mark.gpu
U = (0.1, -0.05, 0.08)


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    _abi.load()


def _run(n, tau, data, calls, **kw):
    phi0, R, seed = data
    sim = LBM(3, list(n), 0.0, [m / 32.0 for m in n], u=U, tau=tau, precision="fp32dev", **kw)
    sim.init(phi0, None, R)
    for c in calls:
        sim.step(c)
    out = [sim.get_state().clone(), sim.macro()]
    sim.adjoint_seed(seed)
    for c in calls:
        sim.adjoint_step(c)
    gphi, _, gR = sim.adjoint_grads(want_grad=False, want_R=True)
    sim.close()
    return out + [gphi, gR]


@pytest.mark.parametrize("n", [(16, 12, 8), (32, 6, 5), (12, 20, 7), (64, 8, 3), (8, 3, 4), (128, 4, 3), (512, 3, 3), (4, 5, 6), (20, 9, 5), (128, 8, 5),
                               (128, 6, 4), (256, 6, 3), (256, 3, 4), (508, 3, 4), (84, 12, 17), (160, 9, 11), (240, 10, 9), (64, 64, 9)])
@pytest.mark.parametrize("tau", [0.5, 0.8])
@pytest.mark.parametrize("source", [True, False])
def test_staged_everywhere_is_bitwise_the_other_kernels(n, tau, source):
    import torch

    rng = np.random.default_rng(sum(n))
    phi0, R, seed = (torch.from_numpy(rng.standard_normal(int(np.prod(n)))).cuda() for _ in range(3))
    data = (phi0, R if source else None, seed)
    runs = [_run(n, tau, data, [7, 1, 3], flags=_abi.FLAG_STAGING), _run(n, tau, data, [1] * 11, flags=_abi.FLAG_STAGING),
            _run(n, tau, data, [7, 1, 3], flags=_abi.FLAG_STAGING, pdl=False), _run(n, tau, data, [1] * 11, staged=False),
            _run(n, tau, data, [11])]
    for r in runs[1:]:
        for a, b in zip(runs[0], r):
            assert torch.equal(a, b)


# nodes on either side of the lines of the default choice: forward 0.82 M (rows of 256), 1.25 M (128), 2 M (two rows a tile); adjoint
# 0.68 M (256), 0.78 M (100), 0.88 M (84), 1.05 M (60), 2 M (tiles of 400), and two stages only (512)
@pytest.mark.parametrize("n", [(256, 64, 50), (256, 64, 51), (128, 96, 101), (128, 96, 102), (240, 90, 92), (240, 90, 94), (256, 52, 51), (256, 52, 52),
                               (100, 80, 97), (100, 80, 98), (84, 96, 109), (84, 96, 110), (60, 128, 136), (60, 128, 137), (200, 100, 99),
                               (200, 100, 101), (512, 50, 42), (384, 30, 28)])
def test_the_default_choice_does_not_show(n):
    import torch

    rng = np.random.default_rng(sum(n))
    data = [torch.from_numpy(rng.standard_normal(int(np.prod(n)))).cuda() for _ in range(3)]
    for a, b in zip(_run(n, 0.8, data, [2]), _run(n, 0.8, data, [2], staged=False)):
        assert torch.equal(a, b)


def test_staged_small_grid_matches_the_oracle():
    import torch

    n = (32, 12, 6)
    S = int(np.prod(n))
    rng = np.random.default_rng(3)
    phi0, grad = rng.standard_normal(S), rng.standard_normal((3, S))
    sim = LBM(3, list(n), 0.0, [m / 32.0 for m in n], u=U, tau=0.8, precision="fp32dev", flags=_abi.FLAG_STAGING)
    sim.init(torch.from_numpy(phi0).cuda(), torch.from_numpy(grad.ravel()).cuda())
    sim.step(40)
    m = O.Model(3, list(n), 0.0, [k / 32.0 for k in n], U, tau=0.8)
    ref = m.phi(m.step(m.init(phi0, grad, 3), 0, 40))
    assert np.max(np.abs(sim.macro().cpu().numpy() - ref)) < 1e-5 * np.max(np.abs(phi0))
    sim.close()


def test_the_wait_hook_reaches_small_grids_and_unknown_bits_are_refused():
    """A grid that calls of many steps otherwise take in shared memory: with the hook its first launch is a staged one and
    gives up on copies in flight (no fault: a wait of zero length)."""
    import torch

    n = (32, 12, 10)
    sim = LBM(3, list(n), 0.0, [m / 32.0 for m in n], u=U, precision="fp32dev", flags=_abi.FLAG_TEST_EXPIRE_WAIT)
    x = torch.ones(int(np.prod(n)), dtype=torch.float64, device="cuda")
    sim.init(x)
    sim.step(6)
    torch.cuda.synchronize()
    with pytest.raises(LHEError):
        sim.step(1)
    sim.close()
    with pytest.raises(LHEError) as ei:
        LBM(3, list(n), 0.0, [m / 32.0 for m in n], precision="fp32dev", flags=_abi.FLAG_STAGING | 64)
    assert ei.value.status == _abi.ERR_ARG
