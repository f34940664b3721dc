"""GPU: the boundary-node kernels of FP32-deviation boxes change their form with the number of boundary nodes (loads first or
behind their branch, 32 to 128 threads, chained or not): boxes on either side of each line against the oracle, with data of
the exact-solution family and with jets, forward and adjoint."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2410_13165_gb300 import LBM, _abi, build, workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    _abi.load()


def _t(a):
    import torch

    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64).ravel()).cuda()


# boundary nodes: 2D 18,004, 20,004, 120,004 and 140,004; 3D 19,192, 19,984, 57,784, 59,152 and 109,456; 4D 17,680, 27,120,
# 32,896, 39,440 and 85,360; 5D 24,992 and 42,242 (152 SMs: 32 threads up to 19,456; one wave up to 116,736, 58,368, 38,912 and 38,912,
# adjoint 136,192, 107,008, 68,096 and 38,912)
SIZES = [(9000, 4), (10000, 4), (60000, 4), (70000, 4), (96, 96, 4), (98, 98, 4), (168, 168, 4), (170, 170, 4), (232, 232, 4), (14,) * 4, (16,) * 4, (17,) * 4, (18,) * 4,
         (23,) * 4, (8,) * 5, (9,) * 5]


def _hi(n, bc):
    return [(m - 1 if bc == "fullway" else m) / 16.0 for m in n]


@pytest.mark.parametrize("bc", ["fullway", "halfway"])
@pytest.mark.parametrize("n", SIZES)
def test_family_boxes_match_the_oracle(n, bc):
    d = len(n)
    u = ((0.02, 0.04, 0.06, 0.08, 0.1) if bc == "fullway" else (0.01, 0.02, 0.01, 0.02, 0.01))[:d]
    wave = dict(a=[1.0, 0.5], kappa=[(np.pi,) * d, (2.0,) + (-1.0,) * (d - 1)], theta=[0.3, 1.1], b=0.2)
    rng = np.random.default_rng(sum(n))
    S, T = int(np.prod(n)), 3
    phi0, grad, target = rng.normal(size=S), rng.normal(size=(d, S)), rng.normal(size=S)
    m = O.Model(d, list(n), 0.0, _hi(n, bc), u, tau=0.8, R=0.7, bc=bc)
    loss_o, gphi_o, _, ggrad_o = m.gradient(phi0, None, target, T, order=3, grad=grad, wave=m.wave(**wave))
    sim = LBM(d, list(n), 0.0, _hi(n, bc), u=u, tau=0.8, R=0.7, bc=bc, precision="fp32dev")
    sim.init(_t(phi0), _t(grad))
    sim.set_boundary_wave(wave["a"], wave["kappa"], wave["theta"], wave["b"])
    sim.step(T)
    r = sim.macro() - _t(target)
    assert abs(0.5 * float((r * r).sum()) - loss_o) < 1e-5 * loss_o
    f = m.init(phi0, grad, 3)
    for i in range(T):
        f = m.step(f, i, 1, m.wave(**wave))
    ref = m.phi(f)
    assert np.max(np.abs(r.cpu().numpy() + target - ref)) < 1e-5 * np.max(np.abs(ref))
    sim.adjoint_seed(r.contiguous())
    sim.adjoint_step(T)
    gphi, ggrad, _ = sim.adjoint_grads(want_grad=True, want_R=False)
    sim.close()
    assert np.max(np.abs(gphi.cpu().numpy() - gphi_o)) < 1e-5 * np.max(np.abs(gphi_o))
    assert np.max(np.abs(ggrad.cpu().numpy() - ggrad_o.ravel())) < 1e-5 * np.max(np.abs(ggrad_o))


@pytest.mark.parametrize("bc", ["fullway", "halfway"])
@pytest.mark.parametrize("n", [(96, 96, 4), (98, 98, 4), (170, 170, 4), (16,) * 4, (18,) * 4, (8,) * 5])
def test_jets_of_the_family_give_the_family(n, bc):
    """Records and family data take different branches of the same kernel: equal to the rounding of the stored floats."""
    d = len(n)
    u = ((0.02, 0.04, 0.06, 0.08, 0.1) if bc == "fullway" else (0.01, 0.02, 0.01, 0.02, 0.01))[:d]
    F = W.fourier_field(d, 2, 60 + d, 0.0, 1.0)
    a, kap, th = F.wave_params()
    res = []
    for jets in (False, True):
        sim = LBM(d, list(n), 0.0, _hi(n, bc), u=u, R=0.4, bc=bc, precision="fp32dev")
        X = W.node_coords(d, list(n), 0.0, sim.dx, halfway=bc == "halfway")
        sim.init(_t(F.value(X)), _t(F.grad(X)))
        if not jets:
            sim.set_boundary_wave(a, kap, th)
            sim.step(2)
        else:
            for i in range(2):
                pts, toff = sim.boundary_points()
                sim.set_boundary_jet(_t(W.wave_jets(pts, i * sim.dt + toff, u, 0.4, a, kap, th)))
                sim.step(1)
        res.append(sim.macro().cpu().numpy())
        sim.close()
    assert np.max(np.abs(res[0] - res[1])) < 1e-6 * np.max(np.abs(res[0]))
