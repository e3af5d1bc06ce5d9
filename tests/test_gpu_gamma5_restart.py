"""The gamma5 variant in mixed precision where its FP32 shadow recursion loses its
biorthogonality (decided by rounding): a solve that stalls starts over from a good x, so
what converges meets the tolerance and what does not returns an x that is no worse than
the zero guess it began from."""
import numpy as np
import pytest

from oracle.wilson import WilsonOperator
from seeded_inputs import gauge_links, gaussian_source
from tests.gpu_util import true_resid

pytestmark = pytest.mark.gpu


def _solve(dims, eps, seed, kappa, n, mode="plain", **kw):
    from paper_0911_2285_gb300 import Solver
    links = gauge_links(dims, eps, seed)
    op = WilsonOperator(links, kappa, dims)
    b = np.stack([gaussian_source(dims, 100 + i) for i in range(n)])
    # one operator shape: which sources are lost depends on the order of the sums
    args = dict(nev=4, m=12, n1=1, tol=1e-10, maxiter=4000, precision="mixed", k_max=4, gamma5=True, autotune=False)
    with Solver(links, dims, kappa, **{**args, **kw}) as s:
        x, info, _ = s.solve(b, mode=mode, raise_on_fail=False)
    return [(info[j], true_resid(op, b[j], x[j])) for j in range(n)]


@pytest.mark.parametrize("dims,eps,seed,kappa", [((4, 4, 4, 6), 0.6, 3, 0.16), ((4, 4, 4, 6), 0.6, 3, 0.155),
                                                 ((6, 6, 6, 6), 0.3, 5, 0.134), ((8, 8, 8, 8), 0.3, 5, 0.133)])
def test_failed_solves_are_no_worse_than_their_start(dims, eps, seed, kappa):
    for info, r in _solve(dims, eps, seed, kappa, 8):
        assert abs(info["true_resid"] - r) <= 1e-6 * r + 1e-13
        assert r <= 1.0 + 1e-6   # FP32 rounding of the residual it is compared by
        if info["iters"] < 4000:
            assert r <= 1e-10


def test_stalled_solves_converge_after_starting_over():
    """Sources of which the recursion alone loses a third to a half at these kappa; those
    that need more iterations than a stall takes have started over."""
    got = _solve((6, 6, 6, 6), 0.3, 5, 0.13, 8) + _solve((6, 6, 6, 6), 0.3, 5, 0.134, 8)
    done = [info["iters"] for info, r in got if r <= 1e-10]
    assert len(done) >= 12
    assert max(done) > 500
