"""The integer sums and roots of the FP64 path at the ends of their ranges, from
the header compiled for the host, against exact rational arithmetic."""
import ctypes
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

HEADER = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1202_4748_gb300", "csrc",
                      "normal64.cuh")
SOURCE = """
#include "%s"
extern "C" int wide(const double* f, double* out, long n) {
    int finite = 0;
    for (long i = 0; i < n; ++i) {
        double g[19];
        for (int k = 0; k < 19; ++k) g[k] = f[19 * i + k];
        const lbf::WideSum<19> s(g);
        __int128 t = 0;
        for (int k = 0; k < 19; ++k) t += s.add(k);
        out[i] = s.value(t);
        finite += s.finite();
    }
    return finite;
}
// the sum through the fixed-point form where it says it holds, ok[i] = 0 elsewhere
template <class T> static void ranged(const T* f, double* out, int* ok, long n) {
    for (long i = 0; i < n; ++i) {
        T g[19];
        for (int k = 0; k < 19; ++k) g[k] = f[19 * i + k];
        const lbf::FixedSum<T, 19> s(g);
        int64_t t = 0;
        for (int k = 0; k < 19; ++k) t += s.m[k];
        out[i] = (ok[i] = s.in_range()) ? s.value(t) : 0.0;
    }
}
extern "C" void ranged64(const double* f, double* out, int* ok, long n) { ranged(f, out, ok, n); }
extern "C" void ranged32(const float* f, double* out, int* ok, long n) { ranged(f, out, ok, n); }
extern "C" void ranged128(const double* f, double* out, int* ok, long n) {
    for (long i = 0; i < n; ++i) {
        double g[19];
        for (int k = 0; k < 19; ++k) g[k] = f[19 * i + k];
        const lbf::WideSum<19> s(g);
        __int128 t = 0;
        for (int k = 0; k < 19; ++k) t += s.add(k);
        out[i] = (ok[i] = s.in_range()) ? s.value(t) : 0.0;
    }
}
extern "C" void roots(const double* x, double* r, double* q, long n) {
    for (long i = 0; i < n; ++i) {
        r[i] = lbf::n64_sqrt(x[i]);
        q[i] = lbf::n64_inv_sqrt(x[i]);
    }
}
""" % HEADER


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("needs g++")
    d = tmp_path_factory.mktemp("fixed_sums")
    src, so = d / "n.cpp", d / "n.so"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-O2", "-shared", "-fPIC", "-o", str(so), str(src)], check=True)
    return ctypes.CDLL(str(so))


def call(fn, f):
    out = np.empty(len(f))
    n = fn(f.ctypes.data_as(ctypes.c_void_p), out.ctypes.data_as(ctypes.c_void_p), ctypes.c_long(len(f)))
    return n, out


def test_wide_sums_keep_what_a_cancellation_leaves(lib):
    """Each of 19 addends is cut at 2^-121 of the largest one's power of two, and
    the sum is rounded once, ties to even: the rounding of the exact sum itself
    wherever no addend is cut."""
    rng = np.random.default_rng(5)
    n = 20_000
    f = rng.standard_normal((n, 19)) * np.exp(rng.uniform(-300, 300, (n, 1))) * np.exp(rng.uniform(-35, 0, (n, 19)))
    f[:, 10:] = -f[:, :9]                                       # what is left: f[9] and
    f[:, 9] *= np.exp(rng.uniform(-60, 0, n))                   # changes of the last bits
    f[: n // 2, 10] *= 1 + 2.0 ** -50
    f[0], f[1, 1:] = 0.0, 0.0
    f[2] = [1.0] + [2.0 ** -53] + [0.0] * 17                    # ties
    f[3] = [1.0 + 2.0 ** -52] + [2.0 ** -53] + [0.0] * 17
    finite, out = call(lib.wide, f)
    assert finite == n
    for row, o in zip(f.tolist(), out.tolist()):
        exact = sum(map(Fraction, row))
        top = Fraction(max(map(abs, row)))
        off = abs(Fraction(o) - exact)
        assert off <= 19 * Fraction(2) ** -121 * top + Fraction(2) ** -53 * abs(exact)
        if min((abs(v) for v in row if v), default=1.0) > float(top) * 2.0 ** -60:
            assert o == float(exact)
    for bad in (np.inf, -np.inf, np.nan):
        g = f[4:5].copy()
        g[0, 5] = bad
        assert call(lib.wide, g)[0] == 0


def test_roots_over_every_exponent(lib):
    """sqrt rounds like the library's (correctly), 1/sqrt to 0.51 units in the last
    place, from the smallest normal double to the largest: random mantissas, those
    next to squares of 27-bit numbers, and those whose root lies closest to half of
    a last place, N + 1/2 with x the double nearest to its square."""
    rng = np.random.default_rng(6)
    n = 400_000
    mant = rng.uniform(0.5, 1.0, n)
    sq = rng.integers(1 << 26, 1 << 27, n).astype(np.float64) ** 2 * 2.0 ** -54
    half = (rng.integers(1 << 52, 1 << 53, n).astype(np.longdouble) + np.longdouble(0.5)) * np.longdouble(2.0) ** -53
    mant = np.concatenate([mant, sq, np.nextafter(sq, 0), np.nextafter(sq, 1), (half * half).astype(np.float64),
                           0.5 * np.nextafter(1, 2) * np.ones(1), [0.5, np.nextafter(1, 0)]])
    mant = np.where(mant >= 1, 0.5, np.where(mant < 0.5, mant * 2, mant))
    x = np.ldexp(mant, rng.integers(-1021, 1025, mant.size))
    for e in (-1021, -1020, 1023, 1024):
        x = np.concatenate([x, np.ldexp(mant[-3000:], e)])
    x = np.concatenate([x, [np.finfo(float).tiny, np.nextafter(np.finfo(float).tiny, 1), np.finfo(float).max]])
    assert np.all(np.isfinite(x)) and x.min() == np.finfo(float).tiny
    r, q = np.empty(x.size), np.empty(x.size)
    lib.roots(*[v.ctypes.data_as(ctypes.c_void_p) for v in (x, r, q)], ctypes.c_long(x.size))
    np.testing.assert_array_equal(r, np.sqrt(x))
    want = np.sqrt(x.astype(np.longdouble))
    assert np.max(np.abs(q * want - 1)) < 1.1 * 2.0 ** -53


@pytest.mark.parametrize("name,dtype,cut", [("ranged64", np.float64, 57), ("ranged32", np.float32, 57),
                                            ("ranged128", np.float64, 121)])
def test_sums_over_every_exponent(lib, name, dtype, cut):
    """Wherever the sum claims to hold it is within 19 x 2^-cut of the largest
    addend and a rounding of the exact one, at every exponent of the type; the
    ordinary ones (1e-200 to 1e200, FP32 1e-18 up) are all claimed."""
    rng = np.random.default_rng(8)
    n = 30_000
    info = np.finfo(dtype)
    top = rng.integers(info.minexp - info.nmant, info.maxexp + 1, n)
    f = rng.uniform(-1, 1, (n, 19)) * np.exp2(rng.uniform(-80, 0, (n, 19)) * rng.integers(0, 2, (n, 1)))
    f[np.arange(n), rng.integers(0, 19, n)] = rng.uniform(0.5, 1, n) * rng.choice([-1, 1], n)
    f[: n // 3] = np.abs(f[: n // 3])                          # sums that overflow
    f = np.ascontiguousarray(np.ldexp(f, top[:, None]).astype(dtype))
    assert np.all(np.isfinite(f))
    out, ok = np.empty(n), np.empty(n, dtype=np.int32)
    getattr(lib, name)(*[v.ctypes.data_as(ctypes.c_void_p) for v in (f, out, ok)], ctypes.c_long(n))
    big = np.max(np.abs(f.astype(np.longdouble)), axis=1)
    ordinary = (big > (1e-200 if dtype == np.float64 else 1e-18)) & (big < 1e200)
    assert np.all(ok[ordinary]) and not np.all(ok)
    for row, o, held in zip(f.astype(np.float64).tolist(), out.tolist(), ok.tolist()):
        if held:
            exact = sum(map(Fraction, row))
            bound = 19 * Fraction(2) ** -cut * Fraction(max(map(abs, row))) + Fraction(2) ** -53 * abs(exact) * (1 + Fraction(2) ** -50)
            assert np.isfinite(o) and abs(Fraction(o) - exact) <= bound
