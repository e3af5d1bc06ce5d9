"""Reliable updates (one cooperative launch per iteration) on lattices whose sites do
not fill its thread blocks, for every operator and recursion that uses them, with
slots that ask for the update in different iterations: solutions against the
oracle's operator in FP64."""
import numpy as np
import pytest

from oracle.wilson import WilsonOperator
from seeded_inputs import gauge_links, gaussian_source, z2_source
from tests.gpu_util import true_resid

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (6, 3, 5, 7), (4, 6, 8, 10), (8, 8, 8, 8)])
@pytest.mark.parametrize("k", [1, 5])
@pytest.mark.parametrize("kind", ["mixed", "fp64", "evenodd", "evenodd_fp64", "gamma5", "bicgstab"])
def test_solutions_after_reliable_updates(dims, k, kind):
    from paper_0911_2285_gb300 import Solver
    if kind.startswith("evenodd") and any(d % 2 for d in dims):
        pytest.skip("even extents only")
    links = gauge_links(dims, 0.3, 5)
    op = WilsonOperator(links, 0.118, dims)
    src = gaussian_source if kind == "gamma5" else z2_source
    # one source of norm 1e-9: its scalars are far from the others'
    b = np.stack([(1e-9 if j == 2 else 1.0) * src(dims, 900 + j) for j in range(k)])
    args = dict(nev=2, m=8, n1=1, tol=1e-12, maxiter=600, k_max=k, precision="fp64" if "fp64" in kind or kind == "gamma5" else "mixed",
                evenodd=kind.startswith("evenodd"), gamma5=kind == "gamma5", bicgstab=kind == "bicgstab")
    with Solver(links, dims, 0.118, **args) as s:
        x, infos, _ = s.solve(b, mode="plain")
    for j in range(k):
        assert infos[j]["reliable_updates"] >= (1 if args["precision"] == "fp64" else 3)
        assert true_resid(op, b[j], x[j]) <= 1.01e-12
