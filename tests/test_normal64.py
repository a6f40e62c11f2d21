"""The integer Box-Muller of the FP64 path against extended precision.

The header is plain C++ and is compiled here with the host compiler.  R, the
cosine and the sine are formed to about 2^-58 relative and rounded once to
double (at most 2^-53 relative), so each is within 1.1 x 2^-53 of the exact
value over the words' whole range; so are the integer roots and sums beside
them.  The normals' words: random words, words near 0 and near 2^32
(where -ln U is large and tiny), the edges of the table's intervals and of the
octants.  numpy's long double (64-bit mantissa or more) is the exact side.
"""
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
static const lbf::LogEntry T[64] = {LB_LOG_TABLE};
extern "C" void normals(const uint32_t* a, const uint32_t* b, double* r, double* c, double* s, long n) {
    auto tab = [](int i) { return T[i]; };
    for (long i = 0; i < n; ++i) {
        r[i] = lbf::n64_radius(a[i], tab);
        lbf::n64_angle(b[i], c[i], s[i]);
    }
}
extern "C" void roots(const double* x, double* r, double* q, long n) {
    for (long i = 0; i < n; ++i) {
        r[i] = lbf::n64_sqrt(x[i]);
        q[i] = lbf::n64_inv_sqrt(x[i]);
    }
}
template <class T> static int sums(const T* f, double* out, long n) {
    int finite = 0;
    for (long i = 0; i < n; ++i) {
        T g[19];
        for (int k = 0; k < 19; ++k) g[k] = f[19 * i + k];
        const lbf::FixedSum<T, 19> s(g);
        int64_t t = 0;
        for (int k = 0; k < 19; ++k) t += k == 7 ? -s.m[k] : s.m[k];
        out[i] = s.value(t);
        finite += s.finite();
    }
    return finite;
}
extern "C" int sums64(const double* f, double* out, long n) { return sums(f, out, n); }
extern "C" int sums32(const float* f, double* out, long n) { return sums(f, out, n); }
""" % HEADER


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if shutil.which("g++") is None or np.finfo(np.longdouble).nmant < 63:
        pytest.skip("needs g++ and an extended long double")
    d = tmp_path_factory.mktemp("normal64")
    src, so = d / "n.cpp", d / "n.so"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-O2", "-shared", "-fPIC", "-o", str(so), str(src)], check=True)
    return ctypes.CDLL(str(so))


def test_radius_and_angle_are_within_rounding_of_the_exact_values(lib):
    rng = np.random.default_rng(1)
    edges = np.array([k << 25 for k in range(128)] + [k << 29 for k in range(8)], dtype=np.int64)
    edges = np.concatenate([edges + d for d in (-2, -1, 0, 1, 2)]) % (1 << 32)
    wide = np.exp(rng.uniform(0, 22, 200_000)).astype(np.int64)
    w = np.concatenate([rng.integers(0, 1 << 32, 500_000), wide, (1 << 32) - 1 - wide, edges,
                        [0, 1, 2, (1 << 32) - 2, (1 << 32) - 1]]).astype(np.uint32)
    got = [np.empty(w.size) for _ in range(3)]
    ptr = [v.ctypes.data_as(ctypes.c_void_p) for v in (w, w, *got)]
    lib.normals(*ptr, ctypes.c_long(w.size))

    L = np.longdouble
    odd = 2 * w.astype(np.int64) + 1                       # U = odd / 2^33
    below1 = ((1 << 33) - odd).astype(L) / L(2) ** 33      # 1 - U, exact
    ln = np.where(below1 < 0.5, np.log1p(-below1), np.log(odd.astype(L) / L(2) ** 33))
    radius = np.sqrt(-2 * ln)
    octant, t = odd >> 30, odd & ((1 << 30) - 1)
    t = np.where(octant & 1, (1 << 30) - t, t)
    x = t.astype(L) / L(2) ** 30 * (4 * np.arctan(L(1)) / 4)
    swap = ((octant + 1) >> 1) & 1
    co = np.where(swap, np.sin(x), np.cos(x)) * np.where(((octant + 2) >> 2) & 1, -1, 1)
    si = np.where(swap, np.cos(x), np.sin(x)) * np.where(octant >> 2, -1, 1)
    for have, want in zip(got, (radius, co, si)):
        assert np.max(np.abs((have.astype(L) - want) / want)) < 1.1 * 2.0 ** -53


def test_roots_are_within_rounding_of_the_exact_values(lib):
    """0.51 units in the last place, over every exponent of a normal double,
    and the library's value for the rest."""
    rng = np.random.default_rng(2)
    x = np.ldexp(rng.uniform(0.5, 1.0, 300_000), rng.integers(-1000, 1000, 300_000))
    x = np.concatenate([x, rng.uniform(0.5, 2.0, 300_000), [1.0, 4.0, 0.25, 2.0, np.nextafter(1, 0), np.nextafter(4, 5)]])
    r, q = np.empty(x.size), np.empty(x.size)
    p = [v.ctypes.data_as(ctypes.c_void_p) for v in (x, r, q)]
    lib.roots(*p, ctypes.c_long(x.size))
    want = np.sqrt(x.astype(np.longdouble))
    assert np.max(np.abs((r - want) / want)) < 1.1 * 2.0 ** -53
    assert np.max(np.abs(q * want - 1)) < 1.1 * 2.0 ** -53
    x = np.array([0.0, np.inf, np.nan, -1.0, 5e-324])
    lib.roots(*[v.ctypes.data_as(ctypes.c_void_p) for v in (x, r, q)], ctypes.c_long(x.size))
    with np.errstate(all="ignore"):
        np.testing.assert_array_equal(r[:5], np.sqrt(x))
        np.testing.assert_array_equal(q[:5], 1.0 / np.sqrt(x))


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
def test_integer_sums(lib, dtype):
    """Each of 19 values enters to half of 2^-57 of the largest's power of two,
    and the sum is rounded once to double; infinities and NaNs are reported."""
    rng = np.random.default_rng(3)
    n = 20_000
    f = rng.standard_normal((n, 19)) * np.exp(rng.uniform(-30, 30, (n, 1))) * np.exp(rng.uniform(-25, 0, (n, 19)))
    f[: n // 4, 10:] = -f[: n // 4, :9]                    # cancelling
    f[0], f[1, 1:] = 0.0, 0.0
    f = np.ascontiguousarray(f.astype(dtype))
    out = np.empty(n)
    call = lib.sums64 if dtype == np.float64 else lib.sums32
    assert call(f.ctypes.data_as(ctypes.c_void_p), out.ctypes.data_as(ctypes.c_void_p), ctypes.c_long(n)) == n
    sign = np.ones(19)
    sign[7] = -1
    exact = [sum(map(Fraction, row)) for row in (f.astype(np.float64) * sign).tolist()]
    off = np.array([float(abs(Fraction(o) - e)) for o, e in zip(out.tolist(), exact)])
    want = np.array([float(e) for e in exact])
    top = np.max(np.abs(f), axis=1).astype(np.float64)
    assert np.all(off <= 19 * 2.0 ** -57 * top + 2.0 ** -53 * np.abs(want) * (1 + 2.0 ** -50))
    for bad in (np.inf, -np.inf, np.nan):
        g = f[:1].copy()
        g[0, 5] = bad
        assert call(g.ctypes.data_as(ctypes.c_void_p), out.ctypes.data_as(ctypes.c_void_p), ctypes.c_long(1)) == 0
