"""The integer-ALU binary64 operations (csrc/dg_intfp64.cuh), compiled for the host, against
IEEE hardware: the same bits for products, quotients and square roots, special values included."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1609_00098_gb300", "csrc")
SRC = """
#include "dg_intfp64.cuh"
using namespace dg::ifp;
extern "C" void run(long n, const double *a, const double *b, double *m, double *d, double *r)
{
    for (long i = 0; i < n; ++i) {
        m[i] = mul(a[i], b[i]);
        d[i] = div(a[i], b[i]);
        r[i] = root(a[i]);
    }
}
extern "C" void run2(long n, const double *a, const double *b, double *h, int *hok, int *c, int *cok)
{
    for (long i = 0; i < n; ++i) {
        h[i] = half_sum_fast(a[i], b[i]);
        hok[i] = half_sum_ok(a[i], b[i]);
        c[i] = close_fast(a[i], b[i]);
        cok[i] = close_ok(a[i], b[i]);
    }
}
"""


def _compile(d, header_dir, *flags):
    src, so = str(d / "t.cpp"), str(d / "t.so")
    with open(src, "w") as f:
        f.write(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", *flags, "-I", header_dir, src,
                    "-o", so], check=True)
    return ctypes.CDLL(so)


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return _compile(tmp_path_factory.mktemp("intfp64"), CSRC)


# The estimates that the division and the root start from, off by RCP (absolute) and RSQRT
# (relative) on top of their own rounding to FP32.
NUDGED = (("return 1.0f / x;", "return (float)(1.0 / (double)x + RCP);"),
          ("return 1.0f / std::sqrt(x);", "return (float)((1.0 + RSQRT) / std::sqrt((double)x));"))


@pytest.fixture(scope="module", params=[(r, q) for r in (-1, 1) for q in (-1, 1)])
def nudged(request, tmp_path_factory):
    """The operations with both estimates at the ends of the ranges that they are exact for."""
    d = tmp_path_factory.mktemp("intfp64_nudged")
    with open(os.path.join(CSRC, "dg_intfp64.cuh")) as f:
        text = f.read()
    for old, new in NUDGED:
        assert text.count(old) == 1
        text = text.replace(old, new)
    with open(d / "dg_intfp64.cuh", "w") as f:
        f.write(text)
    r, q = request.param
    # 2^-22 and 2^-22.5, less the rounding of the estimate itself (half an FP32 ulp below 1)
    return _compile(d, str(d), f"-DRCP=({r * (2.0 ** -22 - 2.0 ** -25)!r})", f"-DRSQRT=({q * (2.0 ** -22.5 - 2.0 ** -24)!r})")


def _operands(kind):
    r = np.random.RandomState(3)
    n = 400000
    bits = r.randint(0, 1 << 62, n, dtype=np.int64).astype(np.uint64) * np.uint64(4) + np.uint64(1)
    mant = bits & np.uint64((1 << 52) - 1)
    if kind == "sparse":      # significands with few bits at either end: exact results, carries, halves
        k = r.randint(0, 52, n).astype(np.uint64)
        mant = np.where(r.rand(n) < 0.5, mant >> k << k, mant | ((np.uint64(1) << k) - np.uint64(1)))
    if kind == "ends":        # significands near 1 and 2, where the estimates' slack is smallest
        k = (bits >> np.uint64(2)) & np.uint64((1 << 30) - 1)
        mant = np.where(r.rand(n) < 0.5, k, np.uint64((1 << 52) - 1) - k)
    exp = r.randint(0, 2048, n) if kind == "any" else r.randint(960, 1087, n)
    sign = r.randint(0, 2, n).astype(np.uint64) << np.uint64(63)
    x = (sign | (exp.astype(np.uint64) << np.uint64(52)) | mant).view(np.float64)
    if kind == "special":
        sp = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, 2.2250738585072014e-308, 1.7976931348623157e308,
                       1.0, -1.0, 2.0, 0.5, 1.0 + 2.0 ** -52, 2.0 - 2.0 ** -52])
        x = sp[r.randint(0, len(sp), n)]
    return x


def _same_bits(lib, ka, kb):
    a, b = _operands(ka), np.roll(_operands(kb), 7)
    m, d, s = (np.empty_like(a) for _ in range(3))
    p = [x.ctypes.data_as(ctypes.c_void_p) for x in (a, b, m, d, s)]
    lib.run(ctypes.c_long(len(a)), *p)
    with np.errstate(all="ignore"):
        for got, ref in ((m, a * b), (d, a / b), (s, np.sqrt(a))):
            nan = np.isnan(ref)
            assert np.array_equal(np.isnan(got), nan)
            assert np.array_equal(got[~nan].view(np.uint64), ref[~nan].view(np.uint64))


@pytest.mark.parametrize("ka", ["near", "sparse", "any", "special"])
@pytest.mark.parametrize("kb", ["near", "sparse", "any", "special"])
def test_same_bits(lib, ka, kb):
    _same_bits(lib, ka, kb)


@pytest.mark.parametrize("ka", ["near", "sparse", "ends"])
@pytest.mark.parametrize("kb", ["near", "sparse", "ends"])
def test_same_bits_from_the_worst_estimates(nudged, ka, kb):
    _same_bits(nudged, ka, kb)


@pytest.mark.parametrize("ka", ["near", "sparse", "any", "special"])
@pytest.mark.parametrize("kb", ["near", "sparse", "any", "special", "patterns"])
def test_half_sum_and_closeness(lib, ka, kb):
    a = np.abs(_operands(ka))
    r = np.random.RandomState(5)
    if kb == "patterns":  # a few patterns from a, and from the lower end of its binade across it
        u = a.view(np.uint64)
        u = np.where(r.rand(len(a)) < 0.3, u >> np.uint64(52) << np.uint64(52), u)
        a = u.view(np.float64)
        b = (u.view(np.int64) + r.randint(-70, 71, len(a))).view(np.float64)
    else:
        b = np.abs(np.roll(_operands(kb), 7))
    a, b = np.ascontiguousarray(a), np.ascontiguousarray(b)
    h = np.empty_like(a)
    hok, c, cok = (np.empty(len(a), np.int32) for _ in range(3))
    lib.run2(ctypes.c_long(len(a)), *[x.ctypes.data_as(ctypes.c_void_p) for x in (a, b, h, hok, c, cok)])
    with np.errstate(all="ignore"):
        ref, close = 0.5 * (a + b), np.abs(a - b) <= 2.0 ** -48 * a
    hok, cok = hok != 0, cok != 0
    assert np.array_equal(h[hok].view(np.uint64), ref[hok].view(np.uint64))
    assert np.array_equal(c[cok] != 0, close[cok])
    if ka == kb == "near":
        assert hok.all() and cok.mean() > 0.9
    if ka == "near" and kb == "patterns":
        assert cok.mean() > 0.5 and close[cok].any() and not close[cok].all()
