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


# a constant field, one that varies along one axis only, a small signal on a large mean, and a velocity that keeps the
# gradient's weights out of the range of float pairs: few roundings or none are decided by the pairs
@pytest.mark.parametrize("kind", ["constant", "rows", "mean", "slow"])
@pytest.mark.parametrize("d,n", [(2, (61, 53)), (3, (19, 17, 21)), (5, (7, 6, 7, 5, 6))])
def test_undecided_nodes_round_once(d, n, kind):
    import torch

    rng = np.random.default_rng(d)
    S = int(np.prod(n))
    u = (1e-14,) * d if kind == "slow" else (0.1, 0.08, 0.06, 0.04, 0.02)[:d]
    phi0 = {"constant": np.full(S, 1.37), "rows": np.sin(np.arange(S) % n[0] * 2 * np.pi / n[0]),
            "mean": 1.37 + 2.0 ** -rng.integers(10, 40, S) * rng.standard_normal(S), "slow": rng.standard_normal(S)}[kind]
    sim = LBM(d, n, hi=[float(m) for m in n], u=u, tau=0.8, precision="fp32dev")
    t = torch.from_numpy(phi0).cuda()
    v = phi0.reshape(n[::-1])
    r = lambda i, k: np.roll(v, -k, d - 1 - i).ravel()  # noqa: E731
    grad = np.stack([(-r(i, 2) + 8 * r(i, 1) - 8 * r(i, -1) + r(i, -2)) / 12 for i in range(d)])
    sim.init(t)
    got = sim.get_state().cpu().numpy()[: sim.Q * S * 4].view(np.float32).reshape(sim.Q, S)
    w, e, half = np.array(sim.omega), np.array(sim.e, dtype=float), 0.5 * (1 - sim.s)
    want = w[:, None] * (half * ((np.array(u) @ grad)[None] - e @ grad))
    size = abs(half) * (np.abs(np.array(u)) @ np.abs(grad) + np.abs(e) @ np.abs(grad))
    # the differences' own rounding: 24 |phi0| of rounded terms over 12, in each direction
    tol = 16 * 2.0 ** -53 * np.abs(w)[:, None] * (size + 2 * d * abs(half) * np.abs(phi0).max())
    ulp = np.spacing(np.abs(want).astype(np.float32)).astype(np.float64)
    bad = np.abs(got - want) > 0.5 * ulp + tol
    assert not bad.any(), (int(bad.sum()), bad.size)
    sim.close()


def _ms(fn):
    import torch

    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    best = 1e30
    for _ in range(6):
        a.record()
        for _ in range(5):
            fn()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b) / 5)
    return best


@pytest.mark.parametrize("kind", ["constant", "mean", "slow"])
@pytest.mark.parametrize("d,n,limit", [(3, 128, 4.0), (5, 16, 4.0)])
def test_undecided_nodes_cost_like_fp64(d, n, limit, kind):
    """Nodes whose roundings the pairs do not decide take one gradient and a few FP64 operations per population: within a
    small multiple of the FP64 initialisation of the same field (a gradient per population took 8 times as long)."""
    import torch

    x = torch.sin(torch.arange(n ** d, dtype=torch.float64, device="cuda"))
    x = {"constant": 0 * x + 1.37, "mean": 1.37 + 1e-6 * x, "slow": x}[kind]
    ms = []
    for precision in ("fp64", "fp32dev"):
        sim = LBM(d, n, u=(1e-14 if kind == "slow" else 0.05,) * d, tau=0.8, precision=precision)
        sim.init(x)
        ms.append(_ms(lambda: sim.init(x)))
        sim.close()
    assert ms[1] < limit * ms[0], ms
