"""FP64 operator with a site's eight terms on eight threads (few sites and fields) against
the site-per-thread form (more of them): both add the same terms in the same order, so
A, A^+ and residuals agree bit for bit. Lattices with extents of 2 and with site counts
that 16 does not divide, on both sides of the line (304 groups of 32 sites)."""
import numpy as np
import pytest

from tests.gpu_util import random_field, small_problem, true_resid

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,k", [((6, 5, 7, 9), 6), ((9, 9, 7, 5), 4), ((2, 10, 6, 14), 8), ((8, 8, 8, 8), 3),
                                    ((8, 8, 8, 19), 2)])
@pytest.mark.parametrize("dagger", [False, True])
def test_one_field_matches_the_batch(dims, k, dagger):
    from paper_0911_2285_gb300 import Solver
    links, op = small_problem(dims)
    v = np.stack([random_field(op.n, 30 + j) for j in range(k)])
    groups = (op.n // 12 + 31) // 32
    assert groups <= 304 < groups * k
    with Solver(links, dims, 0.12, nev=4, m=12, precision="fp64", k_max=k) as s:
        batch = s.apply(v, dagger=dagger)
        for j in range(k):
            assert np.array_equal(s.apply(v[j], dagger=dagger)[0], batch[j])


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (3, 5, 2, 4), (4, 4, 4, 5)])
def test_pair_drives_a_solve(dims):
    """The operator pair on one slot: the FP64 solver reaches the residual asked for."""
    from paper_0911_2285_gb300 import Solver
    links, op = small_problem(dims)
    b = random_field(op.n, 7)
    with Solver(links, dims, 0.12, nev=2, m=8, precision="fp64", k_max=1, tol=1e-10) as s:
        x, info, _ = s.solve(b, mode="plain")
    assert true_resid(op, b, x[0]) <= 2e-10
