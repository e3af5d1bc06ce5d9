"""FP64 split operator pair where the slots of a batch differ in status (one breaks down
while the others iterate), and its residual form against the site-per-thread one: on both
sides of the line the same terms are added in the same order, so the deflated guesses that
are formed from the residuals agree bit for bit."""
import numpy as np
import pytest

from tests.gpu_util import random_field, small_problem
from tests.test_gpu_failures import breakdown_source, free_links

pytestmark = pytest.mark.gpu


def test_breakdown_of_one_slot_leaves_the_others():
    from paper_0911_2285_gb300 import Solver, lqcd
    dims = (4, 4, 4, 4)
    b = np.stack([random_field(12 * 256, 3), breakdown_source(dims), random_field(12 * 256, 4)])
    with Solver(free_links(dims), dims, 1.0 / 6.0, nev=4, m=12, tol=1e-10, precision="fp64", k_max=3) as s:
        alone = [s.solve(b[j], mode="plain", raise_on_fail=False) for j in (0, 2)]
        for _ in range(10):
            x, info, st = s.solve(b, mode="plain", raise_on_fail=False)
            assert st == lqcd.ERR_BREAKDOWN and info[1]["iters"] == 0 and np.all(x[1] == 0)
            for (xa, ia, _), j in zip(alone, (0, 2)):
                assert ia[0]["iters"] == info[j]["iters"]
                assert np.array_equal(xa[0], x[j])


@pytest.mark.parametrize("dims,k", [((6, 5, 7, 9), 6), ((2, 10, 6, 14), 8), ((8, 8, 8, 19), 2)])
def test_residual_of_one_field_matches_the_batch(dims, k):
    from paper_0911_2285_gb300 import Solver
    links, op = small_problem(dims)
    groups = (op.n // 12 + 31) // 32
    assert groups <= 304 < groups * k
    u = np.stack([random_field(op.n, 60 + j) for j in range(3)])
    b = np.stack([random_field(op.n, 70 + j) for j in range(k)])
    x0 = np.stack([random_field(op.n, 90 + j) for j in range(k)])
    with Solver(links, dims, 0.12, nev=4, m=12, precision="fp64", k_max=k) as s:
        s.eigspace_set(u, u)
        batch = s.deflate(b, x0)
        for j in range(k):
            assert np.array_equal(s.deflate(b[j], x0[j])[0], batch[j])
