"""The FP64 helpers that carry the scalars of every solver (fp64.cuh), called one value per
thread, against numpy: conversions bit for bit over both types' whole ranges, reciprocal,
roots and complex quotient to their error bounds, the breakdown comparison also where
squares leave FP64's range.

Bounds: a third-order step from an FP32 seed (relative error 2^-22 or less) leaves 2^-65, so
the results carry the rounding of the last multiply-add (half a unit) and, for 1/sqrt, of
the product m y (half a unit more): at most one unit from the correctly rounded value. The
quotient takes four rounded factors and a complex product: below 8 2^-53 |a / b|."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "fp64.cuh"
using namespace lqcd;
__global__ void probe(int kind, int n, const double* a, double* out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double x = a[4 * i], y = a[4 * i + 1], z = a[4 * i + 2], w = a[4 * i + 3];
    double r = 0.0, s = 0.0;
    if (kind == 0) r = widen(__uint_as_float((unsigned)__double2loint(x)));
    else if (kind == 1) r = __hiloint2double(0, (int)__float_as_uint(narrow(x)));
    else if (kind == 2) r = rcp_fp64(x);
    else if (kind == 3) r = rsqrt_fp64(x);
    else if (kind == 4) r = sqrt_fp64(x);
    else if (kind == 5) { const double2 q = cdiv_fp64(make_double2(x, y), make_double2(z, w)); r = q.x; s = q.y; }
    else r = abs_at_least(make_double2(x, y), 1e-14, z, w) ? 1.0 : 0.0;
    out[2 * i] = r;
    out[2 * i + 1] = s;
}
extern "C" int run(int kind, int n, const double* a, double* out) {
    double *da = nullptr, *dout = nullptr;
    cudaError_t e = cudaMalloc(&da, 32 * (size_t)n);
    if (e == cudaSuccess) e = cudaMalloc(&dout, 16 * (size_t)n);
    if (e == cudaSuccess) e = cudaMemcpy(da, a, 32 * (size_t)n, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) { probe<<<(n + 127) / 128, 128>>>(kind, n, da, dout); e = cudaGetLastError(); }
    if (e == cudaSuccess) e = cudaMemcpy(out, dout, 16 * (size_t)n, cudaMemcpyDeviceToHost);
    cudaFree(da);
    cudaFree(dout);
    return (int)e;
}
"""


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    from paper_0911_2285_gb300 import build
    d = tmp_path_factory.mktemp("fp64")
    (d / "probe.cu").write_text(SOURCE)
    so = os.path.join(d, "probe.so")
    subprocess.run([build._nvcc(), *build.ARCH, *build.FLAGS, "-I", build.CSRC, "-shared", "-o", so, str(d / "probe.cu")],
                   check=True, capture_output=True, timeout=300)
    lib = ctypes.CDLL(so)

    def call(kind, *cols):
        n = len(cols[0])
        a = np.zeros((n, 4))
        for j, c in enumerate(cols):
            a[:, j] = c
        out = np.zeros((n, 2))
        ptr = lambda v: v.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
        assert lib.run(kind, n, ptr(a), ptr(out)) == 0
        return out
    return call


def _any_double(rng, n, lo, hi):
    """Random signs, mantissas and exponent fields lo..hi (0: subnormals, 2047: inf and NaN)."""
    m = rng.integers(0, 1 << 52, n, dtype=np.uint64)
    e = rng.integers(lo, hi + 1, n).astype(np.uint64)
    s = rng.integers(0, 2, n).astype(np.uint64)
    return ((s << np.uint64(63)) | (e << np.uint64(52)) | m).view(np.float64)


def _units(got, ref):
    """Distance in units of the last place (same sign, finite)."""
    return np.abs(got.view(np.int64) - ref.view(np.int64))


def test_widen_is_exact(probe):
    rng = np.random.default_rng(1)
    f = np.concatenate([rng.integers(0, 1 << 32, 1 << 18, dtype=np.uint64).astype(np.uint32),
                        np.array([0, 0x80000000, 1, 0x80000001, 0x007fffff, 0x00800000, 0x7f7fffff, 0x7f800000,
                                  0xff800000, 0x7fc00000, 0x7f800001], dtype=np.uint32)])
    x = f.view(np.float32)
    got = probe(0, f.astype(np.uint64).view(np.float64))[:, 0]
    with np.errstate(invalid="ignore"):
        ref = x.astype(np.float64)
    nan = np.isnan(x)
    assert np.all(np.isnan(got[nan]))
    assert np.array_equal(got[~nan].view(np.int64), ref[~nan].view(np.int64))


def test_narrow_rounds_to_nearest_even(probe):
    rng = np.random.default_rng(2)
    # FP32 numbers of every size and the midpoints between neighbours, with one unit of FP64 either way
    f = np.abs(rng.integers(0, 0x7f800000, 1 << 16).astype(np.uint32).view(np.float32).astype(np.float64))
    sub = rng.integers(0, 0x00900000, 1 << 15).astype(np.uint32)
    lo = sub.view(np.float32).astype(np.float64)
    hi = (sub + 1).astype(np.uint32).view(np.float32).astype(np.float64)
    n = rng.integers(0x00800000, 0x7f7fffff, 1 << 16).astype(np.uint32)
    nlo, nhi = n.view(np.float32).astype(np.float64), (n + 1).astype(np.uint32).view(np.float32).astype(np.float64)
    mid = np.concatenate([(lo + hi) / 2, (nlo + nhi) / 2])
    top = float(np.finfo(np.float32).max) + 2.0 ** 103   # halfway to 2^128
    edge = np.array([0.0, 2.0 ** -150, 2.0 ** -149, 1.5 * 2.0 ** -149, 2.0 ** -126, 2.0 ** -126 - 2.0 ** -150,
                     float(np.finfo(np.float32).max), top, 2.0 ** 128, 1e300, np.inf, 5e-324, 1e-60, 1e-310, 0.1, 1.0])
    mags = np.concatenate([f, lo, mid, np.nextafter(mid, 0.0), np.nextafter(mid, np.inf), edge, np.nextafter(edge, 0.0),
                           np.abs(_any_double(rng, 1 << 16, 0, 2046)), np.abs(_any_double(rng, 1 << 16, 870, 1152))])
    x = np.concatenate([mags, -mags])
    with np.errstate(over="ignore", under="ignore"):
        ref = x.astype(np.float32)
    got = probe(1, x)[:, 0].view(np.uint64).astype(np.uint32)
    assert np.array_equal(got, ref.view(np.uint32))
    nan = np.array([np.nan, -np.nan, np.uint64(0x7ff0000000000001).view(np.float64)])
    assert np.all(np.isnan(probe(1, nan)[:, 0].view(np.uint64).astype(np.uint32).view(np.float32)))


def test_reciprocal_and_roots(probe):
    rng = np.random.default_rng(3)
    edge = np.array([2.0 ** -959, 2.0 ** -958, 2.0 ** 958, 2.0 ** 959, 1.0, np.nextafter(1.0, 0), np.nextafter(2.0, 0),
                     4.0, np.nextafter(4.0, 0), 1e-300, 1e300])
    a = np.concatenate([np.abs(_any_double(rng, 1 << 17, 3, 2043)), edge])
    wide = np.longdouble
    assert _units(probe(2, a)[:, 0], 1.0 / a).max() <= 1
    assert _units(probe(2, -a)[:, 0], -1.0 / a).max() <= 1
    assert _units(probe(3, a)[:, 0], (1 / np.sqrt(a.astype(wide))).astype(np.float64)).max() <= 1
    assert _units(probe(4, a)[:, 0], np.sqrt(a)).max() <= 1
    special = np.array([0.0, np.inf, 5e-324, 1e-310])
    assert np.array_equal(probe(4, special)[:, 0], np.sqrt(special))
    assert np.isnan(probe(4, np.array([np.nan, -1.0]))[:, 0]).all()


def test_complex_quotient(probe):
    rng = np.random.default_rng(4)
    n = 1 << 17
    a = rng.standard_normal((2, n)) * 10.0 ** rng.uniform(-20, 20, n)
    b = rng.standard_normal((2, n)) * 10.0 ** rng.uniform(-260, 260, n)
    b[1, ::3] *= 10.0 ** rng.uniform(-30, 0, len(b[1, ::3]))
    q = probe(5, a[0], a[1], b[0], b[1])
    A, B = [v.astype(np.longdouble) for v in a], [v.astype(np.longdouble) for v in b]
    big = np.maximum(np.abs(B[0]), np.abs(B[1]))   # scaled by a power of two, so that squares stay in range
    e = np.ldexp(np.longdouble(1), -np.frexp(big)[1].astype(np.int32))
    br, bi = B[0] * e, B[1] * e
    d = br * br + bi * bi
    ref = [(A[0] * br + A[1] * bi) / d * e, (A[1] * br - A[0] * bi) / d * e]
    mag = np.maximum(np.abs(ref[0]), np.abs(ref[1]))
    err = np.maximum(np.abs(q[:, 0] - ref[0]), np.abs(q[:, 1] - ref[1])) / mag
    assert float(err.max()) <= 8 * 2.0 ** -53


def test_breakdown_comparison_over_the_whole_range(probe):
    """|z| >= 1e-14 s1 s2 with |z| a little above and below the line, and zero."""
    rng = np.random.default_rng(5)
    n = 1 << 16
    p = rng.uniform(-290, 290, n)                        # 1e-14 s1 s2 = 10^p (every factor in range)
    s1 = 10.0 ** (p / 2)
    s2 = 10.0 ** (p / 2 + 14)
    t = 1e-14 * s1 * s2
    c = rng.uniform(0.1, 0.99, n)
    s = np.sqrt(1 - c * c)
    for f, want in ((1 + 1e-9, 1.0), (1 - 1e-9, 0.0), (1e-40, 0.0), (1e10, 1.0)):
        x, y = f * t * c, f * t * s
        ok = (np.abs(x) > 1e-300) & (np.abs(y) > 1e-300) & np.isfinite(x) & np.isfinite(y)
        assert np.all(probe(6, x[ok], y[ok], s1[ok], s2[ok])[:, 0] == want)
    zero = np.zeros(4)
    assert np.all(probe(6, zero, zero, np.array([1.0, 1e-80, 1e-100, 1e100]), np.ones(4))[:, 0] == 0.0)
    assert np.all(probe(6, np.full(2, np.nan), np.zeros(2), np.ones(2), np.ones(2))[:, 0] == 0.0)
