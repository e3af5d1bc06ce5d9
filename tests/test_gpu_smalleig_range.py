"""Small eigen-solver on matrices with entries whose squares leave FP64's range (a column
whose part below the diagonal is 1e-170, or subnormal, beside entries near 1): backward
error of the right and left vectors as for any other matrix, n 2^-52 times a small factor."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [3, 12, 33, 80])
@pytest.mark.parametrize("tiny", [1e-150, 1e-170, 1e-250, 5e-324])
def test_tiny_entries_below_the_diagonal(n, tiny):
    from paper_0911_2285_gb300 import small_eig
    rng = np.random.default_rng(n)
    c = np.triu(0.05 * (rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))), 1)
    c += np.diag(np.linspace(1.0, 3.0, n) * np.exp(0.3j * np.arange(n)))
    for j in range(0, n - 2, 5):
        c[j + 2:, j] = tiny * rng.choice([1.0, -1.0], n - j - 2)   # nothing on the subdiagonal itself
    lam, y, z = small_eig(c)
    bound = 8 * n * 2.0 ** -52 * np.linalg.norm(c)
    assert np.all(np.isfinite(lam))
    assert np.max(np.linalg.norm(c @ y - y * lam, axis=0)) <= bound
    zn = z / np.linalg.norm(z, axis=0)
    assert np.max(np.linalg.norm(c.conj().T @ zn - zn * np.conj(lam), axis=0)) <= bound
    ref = np.linalg.eigvals(c)
    assert max(np.min(np.abs(ref - v)) for v in lam) <= 1e-8
