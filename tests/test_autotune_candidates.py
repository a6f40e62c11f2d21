"""What the autotuner times, without a GPU: no kernel twice."""
import pytest

import synth


@pytest.mark.parametrize("kw,precision", [(dict(), "fp64"), (dict(tau=0.8), "fp32"), (dict(tau=0.8), "fp64"),
                                          (dict(tau=[1.0] * 18 + [1.1]), "fp32")])
def test_one_row_per_z_chunk_where_every_row_runs_the_split_step(kw, precision):
    from paper_1202_4748_gb300 import autotune
    rows = autotune.variants("D3Q19")
    systems = [synth.system("D3Q19", n=16), synth.system("D3Q19", n=24, **kw)]
    got = [rows[i] for i in autotune.candidates(systems, precision)]
    assert sorted(r[2] for r in got) == sorted({r[2] for r in rows})
    for r in got:                                              # the row names what runs where one does
        split = [x for x in rows if x[2] == r[2] and x[:2] == (16, 8) and x[3:] == (4, 0, 0, 1)]
        assert not split or r == split[0]


@pytest.mark.parametrize("lattice,precision", [("D3Q19", "fp32"), ("D2Q9", "fp32"), ("D2Q9", "fp64")])
def test_all_rows_elsewhere(lattice, precision):
    from paper_1202_4748_gb300 import autotune
    systems = [synth.system(lattice, n=16, tau=[7.0] * (4 if lattice == "D3Q19" else 3) + [1.0] * 15)]
    assert autotune.candidates(systems, precision) == list(range(len(autotune.variants(lattice))))
