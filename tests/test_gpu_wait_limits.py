"""Bounded waits that run out: with a limit far below a copy's latency the kernels give up,
the call reports LQCD_ERR_TIMEOUT, and the calls that follow (default limit) are right."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SHORT = 1   # cycle


@pytest.fixture
def short_waits():
    from paper_0911_2285_gb300 import lqcd
    L = lqcd.lib()

    def on(yes):
        assert L.lqcd_set_wait_limit(SHORT if yes else 0) == lqcd.OK
    yield on
    on(False)


def test_staged_inner_products(short_waits):
    """Fields larger than L2, so that the copies come from memory and a full ring has to be
    waited for; they land before the blocks exit, none in the next call's stages."""
    import torch
    from paper_0911_2285_gb300 import lqcd
    n = 12 * 16 ** 3 * 32
    g = torch.Generator(device="cuda").manual_seed(3)
    X = torch.view_as_complex(torch.randint(-3, 4, (40, n, 2), device="cuda", generator=g).float())
    Y = X[5:13].clone()
    ref = (X.to(torch.complex128).conj() @ Y.to(torch.complex128).T).cpu().numpy()
    for _ in range(3):
        short_waits(True)
        with pytest.raises(lqcd.LQCDError) as e:
            lqcd.field_dots(X, Y, path=1)
        assert e.value.status == lqcd.ERR_TIMEOUT
        short_waits(False)
        c, _ = lqcd.field_dots(X, Y, path=1)
        assert np.array_equal(c, ref)


def _deflated_solver(**kw):
    from paper_0911_2285_gb300 import Solver
    from seeded_inputs import WORKLOADS, workload_links
    w = WORKLOADS["16^3x32"]
    n = 12 * int(np.prod(w["dims"]))
    s = Solver(workload_links("16^3x32"), w["dims"], w["kappa"], nev=8, m=64, n1=1, n_def_max=60, maxiter=2000,
               precision="mixed", k_max=1, autotune=False, **kw)
    rng = np.random.default_rng(8)
    u = rng.standard_normal((40, n, 2)).view(np.complex128)[..., 0] / np.sqrt(2 * n)
    s.eigspace_set(u, u)
    b = rng.standard_normal((n, 2)).view(np.complex128)[..., 0]
    return s, b


def test_deflation_reports_the_timeout_and_keeps_the_guess(short_waits):
    import ctypes
    from paper_0911_2285_gb300 import lqcd
    s, b = _deflated_solver(tol=1e-10)
    with s:
        good = s.deflate(b, np.zeros_like(b))
        x0 = np.zeros_like(b)
        short_waits(True)
        ptr = lambda a: a.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
        assert lqcd.lib().lqcd_deflate(s._h, 1, ptr(b), ptr(x0), 0) == lqcd.ERR_TIMEOUT
        assert "operator" not in lqcd.last_error()
        short_waits(False)
        assert np.all(x0 == 0)
        assert np.array_equal(s.deflate(b, x0), good)
        # nothing is left for the next call to report
        assert s.solve(b, mode="deflated")[1][0]["true_resid"] <= 1e-10


def test_growth_reports_the_timeout_and_keeps_the_space(short_waits):
    """An eigBiCG request whose Ritz vectors are appended with a short limit: the space
    stays as it was, the request itself finishes, and the next one grows the space."""
    import torch
    from paper_0911_2285_gb300 import lqcd
    s, b = _deflated_solver(tol=1e-3)
    with s:
        x = np.zeros_like(b)
        t = s.submit(b, x, mode="eigbicg")
        s.progress(wait=True)          # admitted: deflated guess and first iterations
        torch.cuda.synchronize()
        short_waits(True)
        with pytest.raises(lqcd.LQCDError) as e:
            for _ in range(200):
                s.progress(wait=True)
        assert e.value.status == lqcd.ERR_TIMEOUT
        assert s.eigspace_size() == 40
        short_waits(False)
        done = False
        for _ in range(200):
            s.progress(wait=True)
            done, info, status = s.poll(t)
            if done:
                break
        assert done and status == lqcd.OK and info["true_resid"] <= 1e-3
        assert s.eigspace_size() == 40
        s.solve(b, mode="eigbicg")
        assert s.eigspace_size() > 40


@pytest.mark.parametrize("variant", [{}, {"evenodd": True}, {"precision": "fp64"}])
def test_reliable_update_barrier(short_waits, variant):
    """The grid barriers of a small lattice's reliable update: the solve reports the
    timeout, and the next one gives the bits of the one before."""
    from paper_0911_2285_gb300 import Solver, lqcd
    from seeded_inputs import z2_source
    from tests.gpu_util import small_problem
    dims = (8, 8, 8, 8)
    links, _ = small_problem(dims)
    b = np.stack([z2_source(dims, 60 + j) for j in range(3)])
    with Solver(links, dims, 0.12, nev=4, m=12, tol=1e-10, k_max=3, autotune=False, **variant) as s:
        good = s.solve(b, mode="plain")[0]
        for mode in ("plain", "eigbicg" if variant == {"precision": "fp64"} else "plain"):
            short_waits(True)
            st = s.solve(b, mode=mode, raise_on_fail=False)[2]
            assert st == lqcd.ERR_TIMEOUT
            short_waits(False)
            assert np.array_equal(s.solve(b, mode="plain")[0], good)
