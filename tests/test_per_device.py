"""Values kept per device (kernel attributes): every device gets its own, a failed
one is tried again, and threads may ask at once.  The header is plain C++; and no
launcher keeps such a thing in a flag for the whole process."""
import ctypes
import glob
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1202_4748_gb300", "csrc")
SOURCE = """
#include <thread>
#include <vector>
#include "%s"
static lbf::PerDevice P;
static std::atomic<int> calls[128];
extern "C" int ask(int device, int value) {
    return P.get(device, [&] { calls[device & 127]++; return value; });
}
extern "C" int count(int device) { return calls[device & 127]; }
extern "C" int storm() {                       // 8 threads, 64 devices: everyone sees the device's value
    static lbf::PerDevice Q;
    std::atomic<int> bad{0};
    std::vector<std::thread> t;
    for (int k = 0; k < 8; ++k)
        t.emplace_back([&] {
            for (int r = 0; r < 1000; ++r)
                for (int d = 0; d < 64; ++d)
                    if (Q.get(d, [&] { return d %% 2 ? 1 : -1; }) != (d %% 2 ? 1 : -1)) bad++;
        });
    for (auto& x : t) x.join();
    return bad;
}
""" % os.path.join(CSRC, "per_device.h")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("needs g++")
    d = tmp_path_factory.mktemp("per_device")
    src, so = d / "n.cpp", d / "n.so"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O2", "-pthread", "-shared", "-fPIC", "-o", str(so), str(src)], check=True)
    return ctypes.CDLL(str(so))


def test_each_device_once(lib):
    assert [lib.ask(0, 1), lib.ask(0, -1), lib.count(0)] == [1, 1, 1]
    assert [lib.ask(1, -1), lib.ask(1, 1), lib.count(1)] == [-1, -1, 1]
    assert [lib.ask(2, 0), lib.ask(2, 0), lib.ask(2, 1), lib.ask(2, 0), lib.count(2)] == [0, 0, 1, 1, 3]
    for d in (-1, 64, 100):                                    # no such slot: asked every time
        assert [lib.ask(d, 1), lib.ask(d, -1)] == [1, -1]
    assert lib.storm() == 0


def test_no_launcher_keeps_an_attribute_for_the_whole_process():
    for path in glob.glob(os.path.join(CSRC, "*.c*")) + glob.glob(os.path.join(CSRC, "*.h")):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        assert not re.search(r"\bstatic\s+(bool|int)\s+\w+\s*=", text), path
