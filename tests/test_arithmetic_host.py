"""Scalar arithmetic of the kernels that stands in for single instructions, taken
from the sources as text and compiled for the host: precision changes by bits
(common.cuh) against the conversions, and quotients by a reciprocal and the
remainder (blas.cu, api.cu; Markstein's method) against division."""
import ctypes
import os
import re
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1912_06934_gb300", "csrc")

SHIMS = r"""
#include <cmath>
#include <cstdint>
#include <cstring>
#define __device__
#define __forceinline__ inline
#define __noinline__ __attribute__((noinline))
template <typename A, typename B> static A as(B v) { A a; memcpy(&a, &v, sizeof(a)); return a; }
static unsigned __float_as_uint(float v) { return as<unsigned>(v); }
static float __uint_as_float(unsigned v) { return as<float>(v); }
static long long __double_as_longlong(double v) { return as<long long>(v); }
static int __double2hiint(double v) { return (int)(as<unsigned long long>(v) >> 32); }
static double __hiloint2double(int h, int l) {
    return as<double>(((unsigned long long)(unsigned)h << 32) | (unsigned)l);
}
"""
CALLS = r"""
extern "C" void widen_all(long n, const float *x, double *y) { for (long i = 0; i < n; ++i) y[i] = widen(x[i]); }
extern "C" void narrow_all(long n, const double *x, float *y) { for (long i = 0; i < n; ++i) y[i] = narrow(x[i]); }
extern "C" void div_all(long n, const double *x, const double *d, double *y) {
    for (long i = 0; i < n; ++i) y[i] = div_by(x[i], Divisor{d[i], 1.0 / d[i], fabs(d[i]) >= LO && fabs(d[i]) <= HI});
}
extern "C" void hess_all(long n, const double *x, const double *dd, double *out) {
    for (long i = 0; i < n; ++i) {
        const double d = dd[i], r = 1.0 / d, gi = x[i], q = gi * r;
        out[i] = HESS;
    }
}
"""


def _between(text, start, end):
    i = text.index(start)
    return text[i:text.index(end, i)]


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    read = lambda f: open(os.path.join(CSRC, f)).read()  # noqa: E731
    common, blas, api = read("common.cuh"), read("blas.cu"), read("api.cu")
    lo, hi = re.search(r"fabs\(d\) >= ([\d.e+-]+) && fabs\(d\) <= ([\d.e+-]+)\};", blas).groups()
    hess = re.search(r"const double y =\s*(fabs\(d\)[^;]*?);", api).group(1).replace("gi[u]", "gi")
    src = SHIMS + _between(common, "__device__ __forceinline__ unsigned long long dbits", "template <typename TO>")
    src += _between(blas, "struct Divisor", "__device__ __forceinline__ Divisor cta_divisor")
    src += _between(blas, "__device__ __forceinline__ double div_by", "constexpr int kScaleRows")
    src += CALLS.replace("LO", lo).replace("HI", hi).replace("HESS", hess)
    d = tmp_path_factory.mktemp("arith")
    (d / "a.cpp").write_text(src)
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-o", str(d / "a.so"),
                           str(d / "a.cpp")])
    return ctypes.CDLL(str(d / "a.so"))


def _call(f, *arrays):
    f(ctypes.c_long(len(arrays[0])), *(ctypes.c_void_p(a.ctypes.data) for a in arrays))


def _floats():
    """Every sign and exponent with short, long and random fractions; all ends of the range."""
    rng = np.random.default_rng(1)
    frac = np.concatenate(([0, 1, 2, 3, 0x3fffff, 0x400000, 0x7ffffe, 0x7fffff], rng.integers(0, 1 << 23, 2000)))
    bits = (np.arange(512, dtype=np.uint32)[:, None] << np.uint32(23)) | frac.astype(np.uint32)[None, :]
    return bits.reshape(-1).view(np.float32)


def _same(a, b):
    nan = np.isnan(b)
    u = {4: np.uint32, 8: np.uint64}[b.itemsize]
    return np.array_equal(np.isnan(a), nan) and np.array_equal(a[~nan].view(u), b[~nan].view(u))


def test_widening_by_bits_is_the_conversion(lib):
    x = _floats()
    y = np.empty(len(x))
    _call(lib.widen_all, x, y)
    with np.errstate(invalid="ignore"):
        assert _same(y, x.astype(np.float64))


def test_narrowing_by_bits_is_the_conversion(lib):
    rng = np.random.default_rng(2)
    f = _floats()
    f = f[~np.isnan(f)]
    base = f.astype(np.float64).view(np.uint64)
    tails = [0, 1, 0x0fffffff, 0x10000000, 0x10000001, 0x1fffffff]  # around a tie, to the next float
    x = np.concatenate([base + np.uint64(t) for t in tails]
                       + [rng.integers(0, 1 << 64, 2000000, dtype=np.uint64)]).view(np.float64)
    y = np.empty(len(x), dtype=np.float32)
    _call(lib.narrow_all, x, y)
    with np.errstate(all="ignore"):
        assert _same(y, x.astype(np.float32))


def _random(rng, n, lo, hi):
    bits = (rng.integers(1023 + lo, 1023 + hi, n).astype(np.uint64) << np.uint64(52)) | \
        rng.integers(0, 1 << 52, n, dtype=np.uint64)
    k = n // 4
    bits[:k] |= np.uint64(0xffffffffff000)      # fractions near 2 ...
    bits[k:2 * k] &= np.uint64(0xfff0000000000fff)  # ... and near 1
    bits |= rng.integers(0, 2, n).astype(np.uint64) << np.uint64(63)
    rng.shuffle(bits)
    return bits.view(np.float64)


@pytest.mark.parametrize("which", ["div_all", "hess_all"])
def test_quotients_are_rounded_as_division(lib, which):
    rng = np.random.default_rng(3)
    n = 2000000
    d = _random(rng, n, -460, 460)
    x = _random(rng, n, -450, 460)  # the remainder's last bit stays above 2^-1074
    y = np.empty(n)
    _call(getattr(lib, which), x, d, y)
    assert _same(y, x / d)


@pytest.mark.parametrize("which", ["div_all", "hess_all"])
def test_quotients_at_the_ends_of_the_range(lib, which):
    rng = np.random.default_rng(4)
    n = 400000
    d = np.concatenate((_random(rng, n, -1022, 1023), [1.0, 3.0, -1e-200, 1e200, np.inf, np.nan, 5e-324] * 8))
    x = np.concatenate((_random(rng, n, -1022, 1023), np.repeat([0.0, 1.0, np.inf, -np.inf, np.nan, 5e-324, 1e308,
                                                                 -2.5], 7)))
    y = np.empty(len(d))
    _call(getattr(lib, which), x, d, y)
    with np.errstate(all="ignore"):
        e = x / d
        fin = np.isfinite(e)
        assert np.array_equal(np.isnan(y), np.isnan(e))
        assert np.array_equal(y[~fin & ~np.isnan(e)], e[~fin & ~np.isnan(e)])
        # a remainder below 2^-1074 is lost: the quotient then has the two roundings of x (1 / d)
        assert np.all(np.abs(y[fin] - e[fin]) <= 2.0 ** -51 * np.abs(e[fin]) + 2.0 ** -1073)


def test_zero_divisor(lib):
    x, d = np.array([1.0, 0.0, -3.0]), np.zeros(3)
    y = np.empty(3)
    _call(lib.div_all, x, d, y)
    assert np.all(y == 0.0)  # a zero norm scales to a zero vector
    _call(lib.hess_all, x, d, y)
    assert np.isinf(y[0]) and np.isnan(y[1]) and np.isinf(y[2])
