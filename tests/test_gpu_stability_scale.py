"""GPU stability maps over the size of the weights and of 1 - s: radii of well-parted spectra to rounding, weights far beyond the
stable range, weights that are not finite, and the time that leftover matrices take."""
import time

import numpy as np
import pytest

from paper_2410_13165_gb300 import _abi, build, model, stability_map

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    _abi.load()


def _reference(d, sigma, nxi, tau):
    """Radius by numpy; the condition of the eigenvalue it belongs to (of a simple one: |x| |y| / |y^H x|); the largest row sum."""
    w, _, e = (np.array(v) for v in model(d, sigma, allow_unstable=True))
    s = 1.0 / tau
    xi = -np.pi + 2 * np.pi * np.arange(nxi) / nxi
    grid = np.stack([g.ravel() for g in np.meshgrid(*[xi] * d, indexing="ij")], 1)
    A = np.exp(-1j * grid @ e.T)[:, :, None] * (np.diag(np.full(len(w), 1 - s)) + s * np.outer(w, np.ones(len(w))))[None]
    lam = np.linalg.eigvals(A)
    g = np.argmax(np.abs(lam).max(1))
    lam, V = np.linalg.eig(A[g])
    k = np.argmax(np.abs(lam))
    try:
        cond = np.linalg.norm(np.linalg.inv(V)[k]) * np.linalg.norm(V[:, k])
    except np.linalg.LinAlgError:
        cond = np.inf
    return np.abs(lam[k]), cond, np.abs(A[g]).sum(1).max()


@pytest.mark.parametrize("tau", [0.5, 0.8, 0.45, 1.2, 1.001, 1.00001, 50.0])
@pytest.mark.parametrize("d,nxi", [(1, 31), (2, 9), (2, 16), (3, 6), (3, 7), (4, 3)])
def test_parted_radii_to_rounding(d, nxi, tau):
    rng = np.random.default_rng(7 * d + nxi)
    S = rng.uniform(-0.6, 0.6, (8, d))
    rho, _ = stability_map(d, S, nxi, tau=tau)
    simple = 0
    for p in range(len(S)):
        want, cond, norm = _reference(d, S[p], nxi, tau)
        # rounding of the matrix times the eigenvalue's condition (of a nearly double one: the square root of rounding)
        tol = min(64 * 2.0 ** -53 * norm * cond, 8 * 2.0 ** -26.5 * max(1.0, want))
        simple += tol < 1e-11
        assert abs(rho[p] - want) <= tol, (S[p], rho[p], want, cond)
    assert simple >= 4


@pytest.mark.parametrize("size", [5.0, 100.0, 900.0, 1e4, 1e7])
@pytest.mark.parametrize("tau", [0.5, 0.8, 1.0, 1.001])
@pytest.mark.parametrize("d,nxi", [(1, 16), (2, 7), (3, 4)])
def test_weights_beyond_the_stable_range(d, nxi, tau, size):
    rng = np.random.default_rng(11 * d)
    S = rng.uniform(0.5, 1.0, (4, d)) * rng.choice([-1.0, 1.0], (4, d)) * size
    rho, _ = stability_map(d, S, nxi, tau=tau)
    for p in range(len(S)):
        want, cond, norm = _reference(d, S[p], nxi, tau)
        assert np.isfinite(rho[p]) or size > 1000  # (+inf: the QR iteration gave up on a badly scaled matrix)
        if np.isfinite(rho[p]) and cond < 1e4:
            assert abs(rho[p] - want) <= 64 * 2.0 ** -53 * norm * cond, (S[p], rho[p], want, cond)


@pytest.mark.parametrize("copies", [1, 300, 1100])
def test_leftover_matrices_one_by_one_and_in_numbers(copies):
    """One matrix of these velocities' is left to the QR route: on the list of such matrices, on a longer one, and among more of
    them than the list holds (when all matrices take the route)."""
    rng = np.random.default_rng(42)
    S = rng.uniform(-0.6, 0.6, (6, 2))
    S[0], S[1], S[2], S[3] = 0.0, 0.5, 0.1, 0.5 - 1e-7
    S[1, 1:] = 0.0
    rho, _ = stability_map(2, np.tile(S, (copies, 1)), 9)
    for p in range(len(S)):
        want, cond, norm = _reference(2, S[p], 9, 0.5)
        tol = min(64 * 2.0 ** -53 * norm * cond, 8 * 2.0 ** -26.5 * max(1.0, want))
        assert np.all(np.abs(rho[p::6] - want) <= tol), (S[p], rho[p], want, cond)


@pytest.mark.parametrize("m4", [float("nan"), float("inf")])
@pytest.mark.parametrize("tau", [0.5, 1.0])
def test_weights_that_are_not_finite_are_not_stable(tau, m4):
    rho, _ = stability_map(2, np.array([[0.1, 0.2], [0.0, 0.0]]), 4, tau=tau, m4=[m4])
    assert np.all(np.isinf(rho))


def _seconds(S, nxi):
    best = 1e30
    for _ in range(4):
        t = time.perf_counter()
        stability_map(3, S, nxi)
        best = min(best, time.perf_counter() - t)
    return best


def test_large_weights_take_no_matrix_by_matrix_route():
    """Velocities of order 100: the roots are as well known, relative to the matrix, as for stable weights; with checks in
    absolute terms all of them took the QR route, a lane in eight to 32 at work (180 times as long)."""
    S = np.random.default_rng(5).uniform(-1, 1, (24, 3))
    assert _seconds(S * 100.0, 12) < 8 * _seconds(S * 0.3, 12)
