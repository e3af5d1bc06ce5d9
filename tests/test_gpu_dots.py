"""FP32 inner-product matrices at the edges of the staged kernel's blocks: 4 x 8 blocks
of C, up to 20 warps, 64-element chunks, three stages or more; and on both sides of the
line to the tensor-core form (8 Y fields: ceil(b/8) a against 252 per 128 x 24 tile).
Small integers have exact products and exact FP32 sums, so any lost, doubled or
misplaced element shows; random fields are held to 32 FP32 additions per lane and 5 over
the warp, (32 + 5 + 2) 2^-24 of sum |x||y| <= |x||y|."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _field(k, n, seed, ints):
    import torch
    g = np.random.default_rng(seed)
    z = (g.integers(-3, 4, (k, n)) + 1j * g.integers(-3, 4, (k, n))) if ints else (
        g.standard_normal((k, n)) + 1j * g.standard_normal((k, n)))
    z = z.astype(np.complex64)
    return z, torch.from_numpy(z).cuda()


@pytest.mark.parametrize("a,b,n", [
    (1, 1, 16), (3, 9, 48), (4, 8, 64), (5, 7, 80), (8, 16, 19456), (20, 4, 9728 + 16), (28, 5, 30000), (40, 17, 50000),
    (79, 8, 20464), (80, 8, 19456), (81, 3, 30000), (84, 24, 4096), (85, 24, 4096), (129, 12, 4096), (512, 2, 160)])
def test_edges(a, b, n):
    from paper_0911_2285_gb300.lqcd import field_dots
    for ints in (True, False):
        x, X = _field(a, n, a, ints)
        y, Y = _field(b, n, 100 + b, ints)
        c, _ = field_dots(X, Y, path=1)
        ref = np.conj(x.astype(np.complex128)) @ y.astype(np.complex128).T
        if ints:
            assert np.array_equal(c, ref)
        else:
            bound = np.outer(np.linalg.norm(x, axis=1), np.linalg.norm(y, axis=1))
            assert np.max(np.abs(c - ref) / bound) <= 39 * 2.0 ** -24
