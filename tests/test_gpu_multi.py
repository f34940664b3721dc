"""GPU: periodic boxes taken several steps per launch give, bit for bit, the state, phi and gradients of one step per
call (which is one step per launch): grids on either side of every line of the rule, minimal and ragged extents (tiles that
stick out, regions that wrap), counts of steps that are and are not multiples of a launch's, every collision form (over a
return of the scaled state), constant and per-site sources, both precisions."""
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


def _run(n, precision, tau, R, Rf, calls, back, phi0, seed, pdl=True):
    import torch

    d = len(n)
    sim = LBM(d, list(n), hi=[m / n[0] for m in n], u=(0.1, 0.05, 0.02)[:d], R=R, tau=tau, precision=precision, pdl=pdl)
    sim.init(phi0, None, Rf)
    out = []
    for k in calls:
        sim.step(k)
        out.append(sim.macro())
    out = [out[-1], sim.get_state()]
    sim.adjoint_seed(seed)
    for k in back:
        sim.adjoint_step(k)
    g, _, gR = sim.adjoint_grads(want_grad=False, want_R=True)
    sim.close()
    return out + [g, gR]


GRIDS = [(3,), (9,), (39,), (40,), (131,), (4096,), (30400,), (30401,), (77825,), (3, 3), (4, 5), (7, 6), (9, 13), (16, 16), (64, 64), (61, 67), (85, 86),
         (33, 7), (300, 5), (156, 156), (157, 155), (258, 259), (270, 270), (271, 272), (500, 333), (430, 420), (1224, 1227),
         (3, 3, 3), (5, 4, 6), (8, 8, 8), (16, 16, 16), (17, 15, 17), (24, 24, 24), (25, 23, 25), (7, 40, 11)]


@pytest.mark.parametrize("n", GRIDS)
@pytest.mark.parametrize("precision", ["fp64", "fp32dev"])
def test_steps_per_launch_do_not_show(n, precision):
    import torch

    rng = np.random.default_rng(sum(n))
    S = int(np.prod(n))
    phi0, seed, Rf = (torch.from_numpy(rng.standard_normal(S)).cuda() for _ in range(3))
    forms = [(0.5, 0.0, None), (0.8, 0.7, None), (1.2, 0.0, Rf), (0.5, 0.3, Rf), (1.0, 0.1, None)]
    for i, (tau, R, F) in enumerate(forms if S < 200000 else forms[:3]):
        steps, back = (53, 17) if S < 200000 else (13, 7)
        one = _run(n, precision, tau, R, F, [1] * steps, [1] * back, phi0, seed)
        for calls, bk, pdl in (([steps], [back], True), ([steps - 11, 4, 7], [2, back - 2], True), ([steps], [back], False)):
            for a, b in zip(one, _run(n, precision, tau, R, F, calls, bk, phi0, seed, pdl)):
                assert torch.equal(a, b), (tau, R, F is not None, calls)
