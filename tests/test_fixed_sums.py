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
