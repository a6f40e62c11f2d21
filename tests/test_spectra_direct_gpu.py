"""Spectra of a side beyond the line FFTs (2,048): direct sums along each axis, for
every system of the batch.  One sample against the oracle's (numpy FFT) of the
populations the device holds, per shell: the bars of the other spectra, 1e-10 of
the shell's sum for C(k) and of the sum of its three spectra for the momentum.
"""
import numpy as np
import pytest

import synth
from oracle import observables as ob
from tests.helpers import params_of

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("coupling,sides,jk", [("guo", (2049, 10), True), ("modeq", (20, 2050), False)])
def test_spectra_by_direct_sums_match_the_oracle(coupling, sides, jk):
    import torch
    if not torch.cuda.is_available():
        raise RuntimeError("GPU tests need CUDA; the library has no CPU fallback")
    import paper_1202_4748_gb300 as lb
    systems = [synth.system("D2Q9", coupling, n=n, a=0.01, kT=1e-4, kappa=0.02, seed=9 + k, system_id=k)
               for k, n in enumerate(sides)]
    ens = lb.Ensemble(systems, precision="fp64", sk_every=1, jk_spectra=jk)
    ens.init(amplitude=0.02)
    ens.step(1)
    for k, s in enumerate(systems):
        f, p = ens.read_fields(k), params_of(s)
        want = [ob.structure_factor(ob.order_parameter(f))]
        if jk:
            want += list(ob.momentum_spectra(f, p))
        nb = min(s["nx"], int(np.ceil(np.sqrt(3) * max(sides) / 2)) + 2)
        b = [ob.bin_shells(w, p.shape, nb) for w in want]
        sk, cnt, ns = ens.structure_factor(k, nb)
        assert ns == 1 and np.array_equal(cnt, b[0][1])
        assert np.all(np.abs(sk - b[0][0]) <= 1e-10 * np.abs(b[0][0])), s["nx"]
        if jk:
            got, cnt2, _ = ens.momentum_spectra(k, nb)
            assert np.array_equal(cnt2, b[0][1])
            total = b[1][0] + b[2][0] + b[3][0]
            for c in range(3):
                assert np.all(np.abs(got[c] - b[1 + c][0]) <= 1e-10 * total), (s["nx"], c)
    ens.close()
