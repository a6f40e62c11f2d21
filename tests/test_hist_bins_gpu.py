"""Histograms of as many bins as the interface allows, sampled through every kernel
that counts (thread, warp and CTA bottoms, several ranges per block, coarse
levels): the counts are the oracle's."""
import numpy as np
import pytest

import synth
from oracle import observables as ob
from tests.helpers import params_of

pytestmark = pytest.mark.gpu

SHAPES = {"D2Q9": [(128, 128, 1), (120, 40, 1), (37, 111, 1)],
          "D3Q19": [(32, 32, 32), (20, 20, 20), (34, 34, 34), (27, 25, 23)]}


@pytest.mark.parametrize("lattice", sorted(SHAPES))
@pytest.mark.parametrize("less", [0, 29])
def test_largest_histograms(lattice, less):
    import torch
    if not torch.cuda.is_available():
        raise RuntimeError("GPU tests need CUDA; the library has no CPU fallback")
    import paper_1202_4748_gb300 as lb
    nbins, rng = lb.LB_MAX_HIST_BINS - less, 0.03
    systems = []
    for k, (nx, ny, nz) in enumerate(SHAPES[lattice]):
        s = synth.system(lattice, n=nx, a=-0.002, kT=1e-4, seed=5 + k, system_id=k)
        s.update(nx=nx, ny=ny, nz=nz)
        systems.append(s)
    e = lb.Ensemble(systems, precision="fp64", obs_every=1, hist_bins=nbins, hist_range=rng)
    e.init(amplitude=0.02)
    e.step(1)
    for k, s in enumerate(systems):
        lv = ob.levels(params_of(s))
        want = ob.sample_histograms(ob.order_parameter(e.read_fields(k)), lv, -rng, rng, nbins)
        for l in range(1, len(lv)):                            # (level 0 has m = 0 by conservation)
            assert np.array_equal(e.histogram(k, l)[0].astype(np.int64), want[l]), (k, l)
    e.close()
