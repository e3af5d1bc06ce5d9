"""Device small dense algebra at the sizes where its warp-sliced loops change: the
restart coefficients of window matrices in the form they have after a restart
(kept Ritz values, coupling arrow, tridiagonal part), and the LU factorisation and
solve behind the oblique deflation, against the oracle and numpy in FP64."""
import numpy as np
import pytest

from oracle.bicg import restart_coefficients
from tests.gpu_util import random_field, small_problem

pytestmark = pytest.mark.gpu


def _window_matrix(m, r, seed):
    """Diagonal of r kept values, coupling row and column r, tridiagonal beyond."""
    rng = np.random.default_rng(seed)
    c = lambda n: (rng.standard_normal(n) + 1j * rng.standard_normal(n)) / np.sqrt(2)  # noqa: E731
    H = np.diag(np.linspace(0.2, 3.0, m) + 0.1 * c(m))
    H[r, :r], H[:r, r] = 0.2 * c(r), 0.2 * c(r)
    for k in range(r, m - 1):
        H[k, k + 1], H[k + 1, k] = 0.3 * c(1)[0], 0.3 * c(1)[0]
    return H


@pytest.mark.parametrize("m,nev", [(3, 1), (17, 8), (32, 10), (33, 10), (40, 10), (63, 16), (64, 16)])
def test_restart_coefficients_of_a_restarted_window(m, nev):
    """Eigenvalues of a well-conditioned matrix: double-float rounding (2^-48) times
    the condition of its eigenvalues (below 1e3 here) stays under 1e-10."""
    from paper_0911_2285_gb300 import restart_coefficients as dev_restart
    H = _window_matrix(m, min(2 * nev, m - 1), 300 + m)
    yc_o, zc_o, lam_o = restart_coefficients(H, nev)
    yc, zc, lam = dev_restart(H, nev)
    assert len(lam) == len(lam_o)
    scale = np.abs(lam_o).max()
    for v in lam_o[:nev]:
        assert np.abs(lam - v).min() <= 1e-10 * scale
    assert np.abs(np.conj(zc.T) @ yc - np.eye(len(lam))).max() <= 1e-6
    assert np.abs(np.conj(zc.T) @ H @ yc - np.diag(lam)).max() <= 1e-6 * scale


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 64, 65, 80])
@pytest.mark.parametrize("k", [1, 5])
def test_deflation_solves_with_lu_factors(n, k):
    """x0 + U_r H^{-1} U_l^H (b - A x0) with a Galerkin matrix near the identity
    (condition below 1e3): FP64 rounding of the LU solve stays under 1e-11."""
    from paper_0911_2285_gb300 import Solver
    dims = (4, 4, 4, 4)
    links, op = small_problem(dims)
    rng = np.random.default_rng(40 + n)
    g = lambda m: rng.standard_normal((m, op.n)) + 1j * rng.standard_normal((m, op.n))  # noqa: E731
    ur = g(n) / np.sqrt(2 * op.n)
    ul = ur + 0.2 * g(n) / np.sqrt(2 * op.n)
    b = np.stack([random_field(op.n, 10 + j) for j in range(k)])
    x0 = 0.1 * np.stack([random_field(op.n, 20 + j) for j in range(k)])
    H = np.conj(ul) @ np.stack([op.apply(u) for u in ur]).T
    r = np.stack([b[j] - op.apply(x0[j]) for j in range(k)])
    ref = x0 + np.linalg.solve(H, np.conj(ul) @ r.T).T @ ur
    with Solver(links, dims, 0.12, nev=4, m=12, n1=1, n_def_max=80, precision="fp64", k_max=3) as s:
        s.eigspace_set(ur, ul)
        x = s.deflate(b, x0)
    assert np.abs(x - ref).max() <= 1e-11 * np.abs(ref).max()
