"""The momentum of a site far below its populations, or of populations below the
normal numbers: observables keep its digits.  One site, so the observable is that site's sum c_i f_i alone; the device's
own populations (read back in full) give the exact value."""
from fractions import Fraction

import numpy as np
import pytest

import synth
from oracle import lattice

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("coupling", ["guo", "modeq"])
@pytest.mark.parametrize("name", ["D2Q9", "D3Q19"])
@pytest.mark.parametrize("drift", [1e-6, 1e-10, 1e-14])
def test_momentum_of_a_site_to_rounding(name, coupling, drift):
    import torch
    if not torch.cuda.is_available():
        raise RuntimeError("GPU tests need CUDA; the library has no CPU fallback")
    import paper_1202_4748_gb300 as lb
    lat = lattice.get(name)
    s = synth.system(name, coupling, n=1, a=-0.002, kT=0.0)
    e = lb.Ensemble([s], precision="fp64", obs_every=1)
    e.init(amplitude=0.0)
    f = np.zeros((lat.q, 1, 1, 1))
    c = lat.c.astype(float)
    f[:, 0, 0, 0] = lat.t * (1.0 + 0.01 + 3.0 * drift * (c @ np.array([0.7, -0.4, 0.3 if name == "D3Q19" else 0.0])))
    e.write_fields(0, f)
    e.step(1)
    _, g = e.observables(0)
    got, pops = g["momentum"], e.read_fields(0).ravel()
    for a in range(2 if name == "D2Q9" else 3):
        terms = [Fraction(int(lat.c[i, a])) * Fraction(float(pops[i])) for i in range(1, lat.q)]
        exact, size = sum(terms), sum(map(abs, terms))
        assert abs(exact) > 0.1 * Fraction(drift)
        # one rounding, and what compensated FP64 sums would leave
        assert abs(Fraction(got[a]) - exact) <= Fraction(2) ** -53 * abs(exact) + Fraction(2) ** -105 * size
    e.close()


@pytest.mark.parametrize("coupling", ["guo", "modeq"])
@pytest.mark.parametrize("name", ["D2Q9", "D3Q19"])
@pytest.mark.parametrize("precision,size", [("fp32", 3e-40), ("fp32", 1e-37), ("fp64", 3e-310), ("fp64", 1e-290)])
def test_momentum_of_subnormal_populations(name, coupling, precision, size):
    import torch
    if not torch.cuda.is_available():
        raise RuntimeError("GPU tests need CUDA; the library has no CPU fallback")
    import paper_1202_4748_gb300 as lb
    lat = lattice.get(name)
    e = lb.Ensemble([synth.system(name, coupling, n=1, a=0.0, kT=0.0)], precision=precision, obs_every=1)
    e.init(amplitude=0.0)
    f = np.zeros((lat.q, 1, 1, 1))
    f[0], f[1], f[4] = 1.0, size, 0.5 * size                   # rest: the reference density; +x, -y
    e.write_fields(0, f)
    e.step(1)
    _, g = e.observables(0)
    got, pops = g["momentum"], e.read_fields(0).ravel()
    for a in range(2):
        exact = sum(Fraction(int(lat.c[i, a])) * Fraction(float(pops[i])) for i in range(1, lat.q))
        assert abs(exact) > Fraction(size) / 4
        # one rounding, at most to a subnormal double
        assert abs(Fraction(got[a]) - exact) <= Fraction(2) ** -53 * abs(exact) + Fraction(2) ** -1075
    e.close()
