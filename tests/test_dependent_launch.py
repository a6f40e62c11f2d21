"""Kernels that start before their predecessor has ended promise nothing false.

A kernel that calls grid_wait() runs while an earlier kernel still writes the
populations or the moment field.  A `const T* __restrict__` parameter or local
tells the compiler that the data does not change for the kernel's whole life,
which licenses loads before the wait and through the read-only path; so only the
records that no kernel writes (systems, work items) may carry it.  Read from the
sources: such a race need not show on any one run.
"""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1202_4748_gb300", "csrc")
CONSTANT = {"sysv", "items"}           # written once, before the context exists


def strip_comments(text):
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)


def body_end(text, at):
    depth = 0
    for i in range(text.index("{", at), len(text)):
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return i
    raise AssertionError("unbalanced braces")


def functions(text, start):
    """(name, text) of the functions whose definition `start` matches."""
    for m in re.finditer(start, text):
        brace = text.find("{", m.end())
        if brace < 0 or ";" in text[m.end():brace]:
            continue
        yield m.group("name"), text[m.start():body_end(text, m.end()) + 1]


def test_no_read_only_promise_across_a_grid_wait():
    waiting, called = [], set()
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = strip_comments(open(path).read())
        for name, body in functions(text, r"__global__\s+void\s+(?:__launch_bounds__\([^)]*\)\s*)?(?P<name>\w+)\("):
            if "grid_wait()" not in body:
                continue
            waiting.append(name)
            promised = set(re.findall(r"const\s+[\w:<> ]+?\*\s*__restrict__\s+(\w+)", body))
            assert promised <= CONSTANT, (name, promised - CONSTANT)
            called |= set(re.findall(r"\b(\w+)<[^;{}()]*>\(", body)) | set(re.findall(r"\b(\w+)\(", body))
    assert {"moments_kernel", "moments_quad_kernel", "collide_march_kernel"} <= set(waiting)
    # the device functions they call make no such promise either
    seen = set()
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cuh"))):
        text = strip_comments(open(path).read())
        for name, body in functions(text, r"__device__ __forceinline__ \w+ (?P<name>\w+)\("):
            if name in called:
                seen.add(name)
                assert not re.search(r"const\s+[\w:<> ]+?\*\s*__restrict__", body), name
    assert "pull_site" in seen
