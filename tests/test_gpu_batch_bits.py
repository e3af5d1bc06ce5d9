"""A source gives the same bits alone and in a batch of its context: every sum is formed
in an order that follows from the lattice and the context, not from the other slots.
Lattices of many 128-site units (so that shares of the work could differ), FP64 and mixed,
sources that need their reliable updates at different iterations."""
import numpy as np
import pytest

from tests.gpu_util import random_field, small_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,precision,variant", [
    ((8, 8, 8, 8), "mixed", {}), ((8, 8, 8, 8), "fp64", {}), ((10, 6, 14, 9), "mixed", {}),
    ((8, 8, 8, 12), "mixed", {"evenodd": True}), ((8, 8, 8, 12), "mixed", {"bicgstab": True}), ((6, 6, 6, 10), "fp64", {})])
def test_batch_equals_alone(dims, precision, variant):
    from paper_0911_2285_gb300 import Solver
    links, op = small_problem(dims)
    b = np.stack([random_field(op.n, 50 + j) for j in range(4)])
    b[1, : op.n // 2] = 0.0   # another convergence history
    with Solver(links, dims, 0.12, nev=4, m=12, precision=precision, k_max=4, tol=1e-9, autotune=False, **variant) as s:
        xb, ib, _ = s.solve(b, mode="plain")
        for j in (0, 1, 3):
            xa, ia, _ = s.solve(b[j], mode="plain")
            assert ia[0]["iters"] == ib[j]["iters"]
            assert np.array_equal(xa[0], xb[j])
