"""Spectra of sides with every kind of factor: even and odd, powers of two,
threes, larger primes (a radix of their own in the line FFT) and 1, in batches.

C(k) and the momentum spectra of one sample against the oracle's (numpy FFT) of
the populations the device holds, per shell: 1e-10 of the shell's sum for C(k)
and of the sum of its three spectra for the momentum (the bars of the spectra).
"""
import numpy as np
import pytest

import synth
from oracle import observables as ob
from tests.helpers import params_of

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lattice,coupling,sides", [
    ("D2Q9", "guo", (64, 37, 22, 45, 2, 1, 30, 96)),
    ("D2Q9", "modeq", (120, 7, 3, 50)),
    ("D3Q19", "guo", (16, 9, 10, 2, 1, 7)),
    ("D3Q19", "modeq", (22, 15, 8, 3)),
])
def test_spectra_of_every_side_match_the_oracle(lattice, coupling, sides):
    import torch
    if not torch.cuda.is_available():
        raise RuntimeError("GPU tests need CUDA; the library has no CPU fallback")
    import paper_1202_4748_gb300 as lb
    systems = [synth.system(lattice, coupling, n=n, a=0.01, kT=1e-4, kappa=0.02, seed=9 + k, system_id=k)
               for k, n in enumerate(sides)]
    ens = lb.Ensemble(systems, precision="fp64", sk_every=1, jk_spectra=True)
    ens.init(amplitude=0.02)
    want = [0.0] * len(sides)
    for _ in range(2):
        ens.step(1)
        for k, s in enumerate(systems):
            f, p = ens.read_fields(k), params_of(s)
            want[k] = want[k] + np.concatenate([ob.structure_factor(ob.order_parameter(f))[None],
                                                ob.momentum_spectra(f, p)])
    for k, s in enumerate(systems):
        shape, nb = params_of(s).shape, max(2, s["nx"])
        nb = min(nb, int(np.ceil(np.sqrt(3) * max(sides) / 2)) + 2)
        sk, cnt, ns = ens.structure_factor(k, nb)
        jk, cnt2, _ = ens.momentum_spectra(k, nb)
        assert ns == 2
        if s["nx"] == 1:                              # one site: no wavevector but 0
            assert cnt.sum() == 0 and np.all(sk == 0) and np.all(jk == 0)
            continue
        b = [ob.bin_shells(w, shape, nb) for w in want[k]]
        assert np.array_equal(cnt, b[0][1]) and np.array_equal(cnt2, b[0][1])
        assert np.all(np.abs(sk - b[0][0]) <= 1e-10 * np.abs(b[0][0])), s["nx"]
        total = b[1][0] + b[2][0] + b[3][0]
        for c in range(3):
            assert np.all(np.abs(jk[c] - b[1 + c][0]) <= 1e-10 * total), (s["nx"], c)
    ens.close()
