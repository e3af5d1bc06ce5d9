"""Contexts side by side on one GPU (own streams, one host thread each): every solve gives
the bits that it gives alone, with reliable updates of one context running among the
kernels of the other."""
import threading

import numpy as np
import pytest

from seeded_inputs import z2_source
from tests.gpu_util import small_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kinds", [("mixed", "fp64"), ("evenodd", "bicgstab")])
def test_solves_beside_another_context(kinds):
    from paper_0911_2285_gb300 import Solver
    solvers, srcs, alone = [], [], []
    try:
        for dims, kind, k in (((4, 4, 4, 4), kinds[0], 1), ((12, 12, 12, 16), kinds[1], 4)):
            links, _ = small_problem(dims)
            s = Solver(links, dims, 0.12, nev=2, m=8, tol=1e-10, k_max=k, autotune=False,
                       precision="fp64" if kind == "fp64" else "mixed", evenodd=kind == "evenodd",
                       bicgstab=kind == "bicgstab")
            b = np.stack([z2_source(dims, 40 + j) for j in range(k)])
            solvers.append(s)
            srcs.append(b)
            alone.append(s.solve(b, mode="plain")[0])
        same = []

        def loop(i, n):
            for _ in range(n):
                same.append(np.array_equal(solvers[i].solve(srcs[i], mode="plain")[0], alone[i]))
        threads = [threading.Thread(target=loop, args=(0, 60)), threading.Thread(target=loop, args=(1, 8))]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        assert len(same) == 68 and all(same)
    finally:
        for s in solvers:
            s.close()
