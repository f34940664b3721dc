"""GPU initialisation in FP32 deviations: every stored float is the FP64 value rounded once, also where some terms lie so
far below the others that float pairs drop their low parts."""
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


# exponents of the gradient and of dt R, and the lattice spacing (the gradient's weight is dx (1 - s) / 2 here)
@pytest.mark.parametrize("eg,er,dx", [(-56, -72, 1.0), (-58, -71, 1.0), (-71, -58, 1.0), (-48, -73, 2.0 ** -6), (-75, -48, 2.0 ** 16),
                                      (-72, -50, 2.0 ** 14)])
@pytest.mark.parametrize("d,n", [(1, (200003,)), (2, (301, 303)), (3, (33, 34, 35))])
def test_terms_far_apart_round_once(d, n, eg, er, dx):
    import torch

    rng = np.random.default_rng(eg * er)
    S = int(np.prod(n))
    u = (0.3, 0.1, 0.05)[:d]
    # (dx exact: hi is n dx)
    sim = LBM(d, n, hi=[m * dx for m in n], u=u, tau=0.8, precision="fp32dev")
    grad = rng.uniform(1.0, 2.0, (d, S)) * rng.choice([-1.0, 1.0], (d, S)) * 2.0 ** eg
    R = rng.uniform(1.0, 2.0, S) * rng.choice([-1.0, 1.0], S) * 2.0 ** er / dx
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a).ravel()).cuda()  # noqa: E731
    sim.init(t(rng.standard_normal(S)), t(grad), t(R))
    got = sim.get_state().cpu().numpy()[: sim.Q * S * 4].view(np.float32).reshape(sim.Q, S)
    w, e, s = np.array(sim.omega), np.array(sim.e, dtype=float), sim.s
    dtR, half = sim.dt * R, 0.5 * sim.dt * (1 - s)
    want = w[:, None] * (dtR + half * ((np.array(u) @ grad)[None] - e @ grad))
    # half a unit of the float, and the rounding of a few FP64 operations on terms of this size (here and there)
    size = np.abs(dtR) + abs(half) * (np.abs(np.array(u)) @ np.abs(grad) + np.abs(e) @ np.abs(grad))
    ulp = np.spacing(np.abs(want).astype(np.float32)).astype(np.float64)
    bad = np.abs(got - want) > 0.5 * ulp + 16 * 2.0 ** -53 * np.abs(w)[:, None] * size
    assert not bad.any(), (int(bad.sum()), bad.size)
    sim.close()
