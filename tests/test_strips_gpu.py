"""The row strips of the D2Q9 modified equilibrium: every strip row gives the
bits of the CTA tiles on shapes where strips, rows, staged quads or the halo
beside a strip end raggedly, alone and batched, in every storage and rate
setting, and one step agrees with the oracle within the FP32 bar (1e-5 of max
|f|) or 1e-12 of it in FP64."""
import numpy as np
import pytest

import synth
from oracle import lbm
from tests.helpers import oracle_state, params_of, rel_err

pytestmark = pytest.mark.gpu

EVEN = [(4, 1), (4, 3), (60, 5), (64, 2), (68, 33), (128, 66), (196, 31)]
ODD = [(1, 1), (2, 2), (3, 5), (31, 9), (33, 17), (63, 65), (65, 8), (131, 34)]


@pytest.mark.parametrize("tau", [1.0, [1.0] * 3 + [0.8, 0.9, 0.9, 1.1, 1.1, 0.7]])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("shapes", [EVEN, ODD])
def test_strips_give_the_bits_of_the_tiles(shapes, precision, tau):
    import torch
    if not torch.cuda.is_available():
        raise RuntimeError("GPU tests need CUDA; the library has no CPU fallback")
    import paper_1202_4748_gb300 as lb
    systems = []
    for k, (nx, ny) in enumerate(shapes):
        s = synth.system("D2Q9", "modeq", n=nx, a=-0.002 + 0.001 * (k % 4), kT=1e-4, tau=tau, seed=50 + k, system_id=k)
        s.update(nx=nx, ny=ny, nz=1)
        systems.append(s)
    rows = lb.kernel_variants("D2Q9")
    strips = [r for r, row in enumerate(rows) if row[5] == 2]
    tiles = rows.index((32, 8, 1, 0, 0, 0, 1))
    assert {rows[r][1] for r in strips} >= {4, 8, 16, 32, 64}

    def run(variant):
        e = lb.Ensemble(systems, precision=precision, variant=variant)
        e.init(amplitude=0.02)
        e.step(3)
        e.sync()
        out = [e.read_fields(k) for k in range(len(systems))]
        e.close()
        return out

    want = run(tiles + 1)
    for v in strips + [-1]:
        got = run(v + 1)
        assert all(np.array_equal(a, b) for a, b in zip(want, got)), rows[v] if v >= 0 else "default"
    e = lb.Ensemble(systems, precision=precision)
    for k, s in enumerate(systems):
        e.write_fields(k, oracle_state(params_of(s), steps=2))
    before = [e.read_fields(k) for k in range(len(systems))]
    e.step(1)
    e.sync()
    for k, s in enumerate(systems):
        want1 = lbm.step(before[k], 0, params_of(s))
        assert rel_err(e.read_fields(k), want1) < (1e-5 if precision == "fp32" else 1e-12), shapes[k]
    e.close()
