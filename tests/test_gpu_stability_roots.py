"""The secular-equation route of the stability map against numpy's eigenvalues of the population-space matrix, where its
choices change: every lane-group size (number of poles), odd and even grids, one and two wave numbers, s = 1 (rank
one), s > 2, weights of zero (|sigma_i| = 1/2) and close to it, equal and zero velocities."""
import numpy as np
import pytest

from paper_2410_13165_gb300 import _abi, build, model, stability_map

pytestmark = pytest.mark.gpu

# A double eigenvalue is known to the square root of rounding only (to LAPACK as well): 8 sqrt(2^-53) relative.
TOL = 8 * 2.0 ** -26.5


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    _abi.load()


def _reference(d, sigma, nxi, tau):
    w, _, e = (np.array(v) for v in model(d, sigma, allow_unstable=True))
    s = 1.0 / tau
    xi = -np.pi + 2 * np.pi * np.arange(nxi) / nxi
    grid = np.stack([g.ravel() for g in np.meshgrid(*[xi] * d, indexing="ij")], 1)
    A = np.exp(-1j * grid @ e.T)[:, :, None] * (np.diag(np.full(len(w), 1 - s)) + s * np.outer(w, np.ones(len(w))))[None]
    return np.abs(np.linalg.eigvals(A)).max(), w.min()


@pytest.mark.parametrize("tau", [0.5, 0.8, 1.0, 0.45, 1.001])
@pytest.mark.parametrize("d,nxi", [(1, 1), (1, 7), (1, 4096), (2, 2), (2, 4), (2, 9), (2, 16), (3, 3), (3, 8), (3, 9), (4, 2), (4, 5)])
def test_radius_matches_numpy(d, nxi, tau):
    rng = np.random.default_rng(40 + d)
    S = rng.uniform(-0.6, 0.6, size=(6, d))
    S[0], S[1], S[2], S[3] = 0.0, 0.5, 0.1, 0.5 - 1e-7
    if d > 1:
        S[1, 1:] = 0.0
    rho, omin = stability_map(d, S, nxi, tau=tau)
    for p in range(len(S)):
        want, low = _reference(d, S[p], nxi, tau)
        assert abs(omin[p] - low) < 1e-15
        assert abs(rho[p] - want) <= TOL * max(1.0, want), (S[p], rho[p], want)
