"""GPU: a Dirichlet run gives the same bits however its steps are grouped into calls, with and without programmatic dependent
launch: the manufactured solution (its source scaled inside the row kernel, formed as a field at the end of a call) and
one block of jets per step (step_jets / adjoint_step_jets against the calls they stand for)."""
import math

import numpy as np
import pytest

from paper_2410_13165_gb300 import LBM, _abi, build, jet_len, workloads as W

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


@pytest.mark.parametrize("precision", ["fp64", "fp32dev"])
@pytest.mark.parametrize("bc", ["fullway", "halfway"])
@pytest.mark.parametrize("d,n", [(1, 9), (2, 13), (3, 9)])
def test_sine_product_in_calls_of_any_size(d, n, bc, precision):
    import torch

    th = [0.3 + 0.2 * i for i in range(d)]
    out = []
    for calls, pdl in (([7], True), ([3, 1, 3], True), ([1] * 7, True), ([7], False)):
        sim = LBM(d, n, -1.0, 1.0, u=(1e-3,) * d, bc=bc, precision=precision, pdl=pdl)
        X = W.node_coords(d, [n] * d, -1.0, sim.dx, halfway=bc == "halfway")
        kw = dict(kappa=[math.pi] * d, theta=th)
        sim.set_boundary_sine_product(**kw)
        sim.init(_t(W.sine_product_value(X, 0.0, **kw)), _t(W.sine_product_grad(X, 0.0, **kw)),
                 _t(W.sine_product_source(X, 0.0, (1e-3,) * d, **kw)))
        for k in calls:
            sim.step(k)
        out.append((sim.macro(), sim.get_state(), torch.tensor(sim.diagnostics()["entropy"])))
        sim.close()
    for o in out[1:]:
        for a, b in zip(out[0], o):
            assert torch.equal(a, b)


@pytest.mark.parametrize("precision", ["fp64", "fp32dev"])
@pytest.mark.parametrize("bc", ["fullway", "halfway"])
@pytest.mark.parametrize("d,n,T", [(1, 8, 4), (2, 11, 5), (3, 7, 3), (2, 11, 0)])
def test_steps_with_jets_in_one_call(d, n, T, bc, precision):
    import torch

    rng = np.random.default_rng(3 * d + T)
    res = []
    for native, pdl in ((True, True), (False, True), (True, False)):
        sim = LBM(d, n, u=(1e-3,) * d, R=0.4, bc=bc, precision=precision, pdl=pdl)
        P, JL = len(sim.boundary_points()[0]), jet_len(d)
        if not res:
            jets = torch.from_numpy(rng.standard_normal((T, P, JL))).cuda()
            phi0, grad, seed = (torch.from_numpy(rng.standard_normal(m * sim.S)).cuda() for m in (1, d, 1))
        sim.init(phi0, grad)
        out = torch.full((T, P, JL), float("nan"), dtype=torch.float64, device="cuda")
        if native:
            sim.step_jets(jets)
        else:
            for i in range(T):
                sim.set_boundary_jet(jets[i])
                sim.step(1)
        got = [sim.macro(), sim.get_state()]
        sim.adjoint_seed(seed)
        if native:
            sim.adjoint_step_jets(out)
        else:
            for i in range(T - 1, -1, -1):
                sim.adjoint_jet_grad(out=out[i])
                sim.adjoint_step(1)
        res.append(got + [out] + list(sim.adjoint_grads(want_grad=True, want_R=False))[:2])
        sim.close()
    for r in res[1:]:
        for a, b in zip(res[0], r):
            assert torch.equal(a, b)
    assert not torch.isnan(res[0][2]).any()
