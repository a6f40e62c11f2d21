"""Block observables of systems whose bottom blocks take each of the summing
paths (a thread, a warp, a CTA, several CTAs per block), alone and batched.

The samples of the device are compared with the oracle's block sums of the
populations the device holds at the same times, to 1e-10 relative (the bar of
every observable); the histogram counts are whole numbers and equal.  Level 0
has m = 0 by conservation: its m moments are rounding on both sides.
"""
import numpy as np
import pytest

import synth
from oracle import observables as ob
from tests.helpers import params_of

pytestmark = pytest.mark.gpu

# sides with their bottom block: thread (27 and 1 sites), warp (225, 1000, 125),
# CTA (2197 = one range), several ranges (15525; 2 ranges per block of 17^3)
SHAPES_2D = [(24, 24, 1), (60, 60, 1), (120, 40, 1), (37, 111, 1), (64, 64, 1), (7, 5, 1)]
SHAPES_3D = [(24, 24, 24), (20, 20, 20), (26, 26, 26), (27, 25, 23), (34, 34, 34), (1, 3, 2), (32, 16, 48)]


@pytest.mark.parametrize("lattice,shapes,alone", [("D2Q9", SHAPES_2D, None), ("D3Q19", SHAPES_3D, None),
                                                  ("D3Q19", SHAPES_3D, 3), ("D2Q9", SHAPES_2D, 1)])
def test_block_sums_of_every_path_match_the_oracle(lattice, shapes, alone):
    import torch
    if not torch.cuda.is_available():
        raise RuntimeError("GPU tests need CUDA; the library has no CPU fallback")
    import paper_1202_4748_gb300 as lb
    shapes = shapes if alone is None else [shapes[alone]]
    systems = []
    for k, (nx, ny, nz) in enumerate(shapes):
        s = synth.system(lattice, n=nx, a=-0.002, kT=1e-4, seed=5 + k, system_id=k)
        s.update(nx=nx, ny=ny, nz=nz)
        systems.append(s)
    nbins, rng = 64, 0.03
    ens = lb.Ensemble(systems, precision="fp64", obs_every=1, hist_bins=nbins, hist_range=rng)
    ens.init(amplitude=0.02)
    lvs = [ob.levels(params_of(s)) for s in systems]
    want = [np.zeros((len(lv), 7)) for lv in lvs]
    hist = [np.zeros((len(lv), nbins + 2), dtype=np.int64) for lv in lvs]
    for _ in range(2):
        ens.step(1)
        for k in range(len(systems)):
            phi = ob.order_parameter(ens.read_fields(k))
            want[k] += ob.sample(phi, lvs[k])
            hist[k] += ob.sample_histograms(phi, lvs[k], -rng, rng, nbins)
    for k in range(len(systems)):
        levels, _ = ens.observables(k)
        got = np.array([[L[f] for f in ob.ACC_FIELDS] for L in levels])
        assert [L["block"] for L in levels] == lvs[k]
        assert np.array_equal(got[:, 0], want[k][:, 0])
        assert np.all(np.abs(got[0, 1:5]) < 1e-12)
        assert np.allclose(got[0, 5:], want[k][0, 5:], rtol=1e-10, atol=0)
        scale = np.abs(want[k][1:]).copy()
        scale[:, 1] = want[k][1:, 3]                  # sum m vanishes: |m| scale
        assert np.all(np.abs(got[1:] - want[k][1:]) <= 1e-10 * scale + 1e-300), (shapes[k], got, want[k])
        for l in range(1, len(levels)):
            assert np.array_equal(ens.histogram(k, l)[0].astype(np.int64), hist[k][l]), (shapes[k], l)
    ens.close()
