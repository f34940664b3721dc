"""GPU initialisation: the stored populations against Eq. (ini-simp) with its collision, in numpy, over the ranges where
the kernels change their arithmetic (float pairs, the FP64 form, differences of phi0 formed on the fly)."""
import numpy as np
import pytest

from paper_2410_13165_gb300 import LBM, _abi, build

pytestmark = pytest.mark.gpu

U = {1: (0.3,), 2: (0.1, 0.05), 3: (0.1, 0.1, 0.1), 4: (0.05, 0.2, 0.08, 0.1), 5: (0.02, 0.04, 0.06, 0.08, 0.1)}
N = {1: (37,), 2: (13, 9), 3: (9, 7, 11), 4: (6, 7, 5, 6), 5: (5, 6, 5, 7, 5)}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    _abi.load()


def _fd(p, n, dx):
    v = p.reshape(n[::-1])
    ax = [len(n) - 1 - i for i in range(len(n))]
    r = lambda i, k: np.roll(v, -k, ax[i])  # noqa: E731
    return np.stack([((-r(i, 2) + 8 * r(i, 1) - 8 * r(i, -1) + r(i, -2)) / (12 * dx)).ravel() for i in range(len(n))])


# smooth, noise, a zero field, rows of zeros beside large values, and magnitudes at both ends of the pairs' range
@pytest.mark.parametrize("kind", ["smooth", "noise", "zero", "sparse", "tiny", "small", "large", "huge"])
@pytest.mark.parametrize("given", [True, False])
@pytest.mark.parametrize("source", [True, False])
@pytest.mark.parametrize("d", [1, 2, 3, 4, 5])
def test_init_state(d, given, source, kind):
    import torch

    n, tau, S = N[d], 0.8, int(np.prod(N[d]))
    rng = np.random.default_rng(17 + d)
    scale = {"tiny": 1e-25, "small": 1e-17, "large": 1e28, "huge": 1e33}.get(kind, 1.0)
    phi0 = (np.sin(np.arange(S) * 0.13) + 1.0 if kind in ("smooth",) else rng.standard_normal(S)) * scale
    if kind == "zero":
        phi0[:] = 0.0
    if kind == "sparse":
        phi0[rng.random(S) < 0.8] = 0.0
    R = rng.standard_normal(S) * scale * 0.3 if source else None
    for prec in ("fp64", "fp32dev"):
        sim = LBM(d, n, hi=[m / n[0] for m in n], u=U[d], tau=tau, precision=prec)
        grad = _fd(phi0, n, sim.dx)
        t = lambda a: None if a is None else torch.from_numpy(np.ascontiguousarray(a).ravel()).cuda()  # noqa: E731
        sim.init(t(phi0), t(grad) if given else None, t(R))
        raw = sim.get_state().cpu().numpy()
        w, e, s = np.array(sim.omega), np.array(sim.e, dtype=float), sim.s
        g = np.zeros(S) if R is None else sim.dt * R
        corr = 0.5 * sim.dt * (1 - s) * ((np.array(U[d]) @ grad)[None] - e @ grad)  # (Q, S)
        size = 0.5 * sim.dt * abs(1 - s) * (np.abs(e) @ np.abs(grad) + np.abs(grad).sum(0)) + np.abs(g)
        if prec == "fp64":
            got, want = raw.view(np.float64).reshape(sim.Q, S), w[:, None] * (phi0 + g + corr)
            # rounding of a few operations on terms of this size (and of the differences, of the values they take)
            tol = 16 * 2.0 ** -53 * np.abs(w)[:, None] * (size + np.abs(phi0)) + 8 * 2.0 ** -53 * np.abs(phi0).max()
            assert np.all(np.abs(got - want) <= tol)
        else:
            got = raw[: sim.Q * S * 4].view(np.float32).reshape(sim.Q, S)
            want = w[:, None] * (g + corr)
            with np.errstate(over="ignore"):
                ulp = np.spacing(np.abs(want).astype(np.float32)).astype(np.float64)
            tol = 0.5 * ulp + 16 * 2.0 ** -53 * np.abs(w)[:, None] * size + 8 * 2.0 ** -53 * np.abs(phi0).max() * np.abs(w).max()
            bad = ~(np.abs(got - want) <= tol)
            assert not bad.any(), (np.argwhere(bad)[:5], got[bad][:5], want[bad][:5])
            h, l = raw[sim.Q * S * 4:].view(np.float32).reshape(S, 2).astype(np.float64).T
            assert np.all(np.abs(h + l - phi0) <= 2.0 ** -48 * np.abs(phi0) + 2.0 ** -149)
        sim.close()
