"""Inner-product matrices large enough for the tensor-core form (3xTF32 tcgen05 MMAs; path 1
takes it where ceil(b/8) a exceeds 252 per 128 x 24 tile): ragged row tiles and groups of Y
fields, few and many K-tiles. Integers are exact in TF32 and their sums in FP32, so that a
lost, doubled or misplaced tile shows; on random fields the FP32-level bounds of the form
(2e-6 of |x| |y|, 1e-6 of a squared norm, where truncation would add up)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _takes_tensor_cores(a, b):
    return -(-b // 8) * a > 252 * -(-a // 128) * -(-b // 24)


def _fields(k, n, seed, ints):
    import torch
    g = torch.Generator(device="cuda").manual_seed(seed)
    z = (torch.randint(-3, 4, (k, n, 2), device="cuda", generator=g).float() if ints
         else torch.randn((k, n, 2), device="cuda", generator=g))
    return torch.view_as_complex(z)


def _ref(X, Y):
    import torch
    out = torch.zeros(X.shape[0], Y.shape[0], dtype=torch.complex128, device="cuda")
    for e in range(0, X.shape[1], 1 << 16):
        out += X[:, e:e + (1 << 16)].to(torch.complex128).conj() @ Y[:, e:e + (1 << 16)].to(torch.complex128).T
    return out.cpu().numpy()


@pytest.mark.parametrize("a,b,n", [(85, 24, 16), (128, 17, 48), (120, 24, 49152 + 16), (200, 47, 3072), (256, 48, 1040),
                                   (127, 72, 30000), (384, 20, 4096), (512, 24, 1600)])
def test_integer_fields_exact(a, b, n):
    from paper_0911_2285_gb300.lqcd import field_dots
    assert _takes_tensor_cores(a, b)
    X, Y = _fields(a, n, 1 + a, True), _fields(b, n, 2 + b, True)
    assert np.array_equal(field_dots(X, Y, path=1)[0], _ref(X, Y))


@pytest.mark.parametrize("a,b,n", [(96, 24, 1572864), (200, 47, 196608), (128, 24, 49152)])
def test_random_fields(a, b, n):
    import torch
    from paper_0911_2285_gb300.lqcd import field_dots
    assert _takes_tensor_cores(a, b)
    X, Y = _fields(a, n, 10 + a, False), _fields(b, n, 20 + b, False)
    c = field_dots(X, Y, path=1)[0]
    nx, ny = (torch.linalg.vector_norm(Z, dim=1, dtype=torch.complex128).real.cpu().numpy() for Z in (X, Y))
    assert np.max(np.abs(c - _ref(X, Y)) / np.outer(nx, ny)) <= 2e-6


def test_norms_without_cancellation():
    """Sums of positive terms only, over many K-tiles: truncation would show undiminished."""
    import torch
    from paper_0911_2285_gb300.lqcd import field_dots
    assert _takes_tensor_cores(96, 96)
    X = _fields(96, 884736, 77, False)
    c = field_dots(X, X, path=1)[0]
    nrm = (X.real.double() ** 2 + X.imag.double() ** 2).sum(1).cpu().numpy()
    assert np.max(np.abs(np.diag(c).real - nrm) / nrm) <= 1e-6
    assert np.max(np.abs(np.diag(c).imag)) <= 1e-6 * nrm.max()
