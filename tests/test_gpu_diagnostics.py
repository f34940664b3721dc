"""GPU diagnostics of a caller's state (set_state) against the sums in numpy: every lattice, both precisions, s = 1, s = 2 and
general s, sizes from a fraction of a block to several passes of the grid, and states with infinities and NaN."""
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


def _sim_and_state(d, n, precision, tau, seed):
    import torch

    sim = LBM(d, n, hi=[m / n[0] for m in n], R=0.7, tau=tau, precision=precision)
    rng = np.random.default_rng(seed)
    if precision == "fp64":
        f = rng.standard_normal((sim.Q, sim.S))
        buf, phi = f.tobytes(), None
    else:
        f, phi = rng.standard_normal((sim.Q, sim.S)).astype(np.float32), rng.standard_normal((sim.S, 2)).astype(np.float32)
        phi[:, 1] *= 2.0 ** -25
        buf = f.tobytes() + phi.tobytes()
    return sim, f, phi, lambda b: torch.frombuffer(bytearray(b), dtype=torch.uint8).cuda(), buf


@pytest.mark.parametrize("tau", [0.5, 0.8, 1.0])
@pytest.mark.parametrize("precision", ["fp64", "fp32dev"])
@pytest.mark.parametrize("d,n", [(1, (7,)), (2, (31, 9)), (3, (70, 61, 53)), (4, (5, 9, 7, 6)), (5, (5, 4, 6, 3, 7))])
def test_diagnostics_of_a_state(d, n, precision, tau):
    sim, f, phi, dev, buf = _sim_and_state(d, n, precision, tau, 5 * d)
    w, s, dtR = np.array(sim.omega)[:, None], sim.s, sim.dt * 0.7
    f = f.astype(np.float64)
    p = f.sum(0) - dtR if precision == "fp64" else phi.astype(np.float64).sum(1)
    back = (f - w * ((s * p + dtR) if precision == "fp64" else dtR)) / (1 - s) if s != 1.0 else f
    ent = (back ** 2 / (2 * w)).sum(0) + (0.0 if precision == "fp64" else 0.5 * p * p)
    for _ in range(2):  # the second call reuses the first one's scratch
        sim.set_state(dev(buf), 0)
        got = sim.diagnostics()
        assert got["ok"] and got["nonfinite"] == 0
        # rounding of S terms added in any order
        assert abs(got["mass"] - p.sum()) <= 2.0 ** -52 * sim.S * np.abs(p).sum()
        assert abs(got["entropy"] - ent.sum()) <= 2.0 ** -52 * (sim.S + 8 * sim.Q) * ent.sum()
        assert abs(got["max_abs"] - np.abs(p).max()) <= 2.0 ** -52 * sim.Q * np.abs(f).max()
    sim.close()


@pytest.mark.parametrize("precision", ["fp64", "fp32dev"])
def test_diagnostics_count_non_finite_values(precision):
    sim, f, phi, dev, buf = _sim_and_state(3, (9, 8, 7), precision, 0.8, 3)
    f[4, 17], f[7, 17], f[2, 400] = np.inf, np.inf, np.nan
    sim.set_state(dev(f.tobytes() + (b"" if phi is None else phi.tobytes())), 0)
    got = sim.diagnostics()
    assert not got["ok"] and got["nonfinite"] == 3
    f[2, 400] = 0.0
    sim.set_state(dev(f.tobytes() + (b"" if phi is None else phi.tobytes())), 0)
    got = sim.diagnostics()
    assert got["nonfinite"] == 2
    if precision == "fp64":
        assert got["mass"] == np.inf and got["max_abs"] == np.inf
    sim.close()
