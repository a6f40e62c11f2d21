"""lb_read_fields leaves the caller's array alone when it cannot read.

The call synchronises, so on a stream that is being captured it returns a CUDA
error (a host-side refusal; nothing runs); the array keeps its contents, and the
context goes on working after the capture has ended.
"""
import ctypes

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lattice,n", [("D2Q9", 96), ("D3Q19", 20)])
def test_failed_read_changes_nothing(lattice, n):
    import torch
    if not torch.cuda.is_available():
        raise RuntimeError("GPU tests need CUDA; the library has no CPU fallback")
    import paper_1202_4748_gb300 as lb
    stream = torch.cuda.Stream()
    e = lb.Ensemble([synth.system(lattice, n=n)], precision="fp32", stream=stream)
    e.init(amplitude=0.02)
    e.step(2)
    e.sync()
    want = e.read_fields(0)
    out = np.full(want.size, 7.25)
    out.view(np.uint8)[::64] = 0xA5
    before = out.copy()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(stream):
        graph.capture_begin(capture_error_mode="relaxed")
        try:
            status = lb.lb_read_fields(e.ctx, 0, out.ctypes.data_as(ctypes.c_void_p))
        finally:
            try:
                graph.capture_end()
            except RuntimeError:
                pass
    assert status == lb.LB_ERR_CUDA
    assert np.array_equal(out.view(np.uint8), before.view(np.uint8))
    lb.lb_read_fields(e.ctx, 0, out.ctypes.data_as(ctypes.c_void_p))      # may report the broken capture once more
    assert np.array_equal(e.read_fields(0), want)
    e.close()
