"""The integer Box-Muller of the FP64 path against extended precision.

The header is plain C++ and is compiled here with the host compiler.  R, the
cosine and the sine are formed to about 2^-58 relative and rounded once to
double (at most 2^-53 relative), so each is within 1.1 x 2^-53 of the exact
value over the words' whole range: random words, words near 0 and near 2^32
(where -ln U is large and tiny), the edges of the table's intervals and of the
octants.  numpy's long double (64-bit mantissa or more) is the exact side.
"""
import ctypes
import os
import shutil
import subprocess

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
