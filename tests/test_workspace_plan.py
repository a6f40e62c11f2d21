"""What lb_workspace_bytes plans, without a GPU."""
import pytest

import synth


def boxes(shapes, lattice="D3Q19", coupling="guo", **kw):
    out = []
    for k, (nx, ny, nz) in enumerate(shapes):
        s = synth.system(lattice, coupling, n=nx, seed=1 + k, system_id=k, **kw)
        s.update(nx=nx, ny=ny, nz=nz)
        out.append(s)
    return out


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("coupling", ["guo", "modeq"])
@pytest.mark.parametrize("shapes", [[(28, 25, 23)], [(28, 25, 23)] * 400, [(27, 25, 23)] * 200, [(16, 16, 16)],
                                    [(64, 64, 64)] * 20, [(24, 24, 24)] * 9])
def test_default_size_covers_every_row_the_default_may_be(precision, coupling, shapes):
    """The default row follows the SMs of the device that is current; a size asked
    for while another device (or none) is current has to do for lb_create."""
    import paper_1202_4748_gb300 as lb
    systems = boxes(shapes, coupling=coupling)
    have = lb.workspace_bytes(systems, precision=precision, obs_every=1)
    for r, row in enumerate(lb.kernel_variants("D3Q19")):
        if row[:2] == (16, 8) and row[3:] == (4, 0, 0, 1) or row[:2] == (32, 8) and row[3:] == (3, 4, 3, 2):
            assert lb.workspace_bytes(systems, precision=precision, obs_every=1, variant=r + 1) <= have, row
    for coup2 in ("modeq", "guo"):
        flat = boxes([(s[0], s[1], 1) for s in shapes], "D2Q9", coup2)
        have2 = lb.workspace_bytes(flat, precision=precision, obs_every=1)
        for r, row in enumerate(lb.kernel_variants("D2Q9")):
            if coup2 == "modeq" and row[0] == 64 and row[5] == 2:
                assert lb.workspace_bytes(flat, precision=precision, obs_every=1, variant=r + 1) <= have2, row


@pytest.mark.parametrize("lattice,n", [("D3Q19", 64), ("D3Q19", 45), ("D3Q19", 2), ("D2Q9", 512), ("D2Q9", 33),
                                       ("D2Q9", 2100)])
def test_momentum_spectra_share_their_transforms_room(lattice, n):
    """Beside what the structure factor needs: the momentum (3 fields), a Laplacian,
    3 complex transforms and 3 accumulators, 104 bytes a site; the half spectra of
    the line FFTs are those transforms, not a region of their own."""
    import paper_1202_4748_gb300 as lb
    s = synth.system(lattice, n=n)
    sites = s["nx"] * s["ny"] * s["nz"]
    a = lb.workspace_bytes([s], precision="fp32", sk_every=5)
    b = lb.workspace_bytes([s], precision="fp32", sk_every=5, jk_spectra=True)
    lines = 16 * 40 * sites // n                       # longer work lists (16 bytes per few lines)
    assert 13 * 8 * sites - 2048 <= b - a <= 13 * 8 * sites + lines // 8 + 8192
