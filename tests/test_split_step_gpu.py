"""The split step (moment pass, then collision columns) of the fully relaxed
FP32 path on D3Q19: the same bits as the one-site kernels on every shape where
its tiles, chunks, rows or quads end raggedly, alone and batched, and one step
against the oracle within the FP32 bar (1e-5 of max |f|)."""
import numpy as np
import pytest

import synth
from oracle import lbm
from tests.helpers import oracle_state, params_of, rel_err

pytestmark = pytest.mark.gpu

def is_split(row):
    return row[:2] == (16, 8) and row[3:] == (4, 0, 0, 1)


EVEN = [(16, 16, 16), (4, 1, 1), (4, 2, 3), (8, 8, 9), (12, 7, 33), (20, 17, 2), (64, 9, 5), (132, 8, 4)]
ODD = [(1, 1, 1), (2, 2, 2), (3, 1, 2), (5, 4, 3), (15, 8, 1), (17, 9, 33), (27, 27, 27), (33, 16, 8), (129, 5, 6)]


@pytest.mark.parametrize("coupling", ["guo", "modeq"])
@pytest.mark.parametrize("shapes", [EVEN, ODD, [(16, 16, 16)], [(45, 50, 37)], [(64, 64, 64)]])
def test_split_rows_give_the_bits_of_the_one_site_kernels(coupling, shapes):
    import torch
    if not torch.cuda.is_available():
        raise RuntimeError("GPU tests need CUDA; the library has no CPU fallback")
    import paper_1202_4748_gb300 as lb
    systems = []
    for k, (nx, ny, nz) in enumerate(shapes):
        s = synth.system("D3Q19", coupling, n=nx, a=-0.002 + 0.001 * (k % 4), kT=1e-4, seed=30 + k, system_id=k)
        s.update(nx=nx, ny=ny, nz=nz)
        systems.append(s)
    rows = lb.kernel_variants("D3Q19")
    one_site = rows.index((16, 8, 16, 6, 0, 0, 1))
    split = [r for r, row in enumerate(rows) if is_split(row)]
    assert split

    def run(variant, chunk):
        e = lb.Ensemble(systems, precision="fp32", variant=variant, graph_chunk=chunk)
        e.init(amplitude=0.02)
        e.step(4)
        e.sync()
        out = [e.read_fields(k) for k in range(len(systems))]
        e.close()
        return out

    want = run(one_site + 1, 0)
    for v in split + [-1]:
        for chunk in (0, 2):
            got = run(v + 1, chunk)
            assert all(np.array_equal(a, b) for a, b in zip(want, got)), (rows[v] if v >= 0 else "default", chunk)
    small = min(range(len(shapes)), key=lambda k: (np.prod(shapes[k]) < 100, np.prod(shapes[k])))
    p = params_of(systems[small])
    if p.n_sites <= 1 << 15:
        e = lb.Ensemble(systems, precision="fp32", variant=split[0] + 1)
        e.write_fields(small, oracle_state(p, steps=2))
        f0 = e.read_fields(small)
        for k in range(len(systems)):
            if k != small:
                e.write_fields(k, lbm.initial_state(params_of(systems[k])))
        e.step(1)
        e.sync()
        assert rel_err(e.read_fields(small), lbm.step(f0, 0, p)) < 1e-5
        e.close()


def test_default_rows_of_small_and_odd_ensembles():
    """Few tiles, or an nx that is not a multiple of 4: the split step; large
    ensembles of even sides keep the paired kernel."""
    import paper_1202_4748_gb300 as lb
    rows = lb.kernel_variants("D3Q19")

    def scheme(n, count, **kw):
        systems = [synth.system("D3Q19", n=n, seed=1 + k, system_id=k, **kw) for k in range(count)]
        e = lb.Ensemble(systems, precision="fp32")
        r = rows[e.kernel_variant()]
        e.close()
        return r

    assert is_split(scheme(16, 1)) and is_split(scheme(64, 1)) and is_split(scheme(27, 40))
    assert scheme(64, 16)[5] == 3 and scheme(64, 32)[:3] == rows[0][:3]
    assert is_split(scheme(16, 1, tau=0.8))
