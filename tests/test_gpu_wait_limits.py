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
