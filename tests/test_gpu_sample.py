"""The synthetic sample generated on the device against the oracle's, bit for
bit: the mask, the chord length and the identity that a saved state carries
(the same geometry handed over as a mask takes the state)."""
import numpy as np
import pytest

from oracle import oracle

pytestmark = pytest.mark.gpu

CASES = [
    # nx, ny, nz, z0, z1, porosity, corr_len, seed, periodic
    (24, 20, 40, 12, 28, 0.65, 3.0, 11, False),
    (33, 29, 50, 2, 48, 0.6, 8.0, 5, False),  # odd lines, the widest slab between open ends
    (128, 96, 100, 20, 81, 0.62, 10.0, 9, False),  # two hash chunks
    (64, 40, 1, 0, 1, 0.5, 2.0, 3, True),  # (nz below 4: refused by both)
    (30, 7, 24, 0, 24, 0.45, 0.0, 2, True),  # no smoothing: many ties, the whole box
    (300, 1, 41, 5, 36, 0.7, 0.6, 8, False),  # one cell along y
    (1, 260, 32, 4, 25, 0.31, 12.0, 17, False),  # one along x
    (16, 12, 40, 8, 30, 0.55, 60.0, 21, False),  # a window of several lines
    (40, 36, 700, 100, 633, 0.66, 5.0, 4, False),  # fewer lines to a block
    (2, 3, 6500, 10, 6400, 0.6, 4.0, 6, False),  # a line too long for a block
    (9, 8, 20, 6, 14, 0.6, 2.0, 7, False),  # too small for the scratch
    (32, 32, 40, 10, 30, 0.0, 3.0, 1, False),
    (32, 32, 40, 10, 30, 1.0, 3.0, 1, False),
    (32, 32, 40, 10, 10, 0.5, 3.0, 1, False),  # an empty slab
    (32, 32, 40, 0, 40, 1.0, 3.0, 1, False),  # between the open ends, all fluid
]


@pytest.mark.parametrize("nx,ny,nz,z0,z1,porosity,corr_len,seed,periodic", CASES)
def test_sample_equals_the_oracles(nx, ny, nz, z0, z1, porosity, corr_len, seed, periodic):
    from paper_1607_02874_gb300 import lbm

    kw = dict(bc=lbm.BC_PERIODIC) if periodic else {}
    if nz < 4:
        with pytest.raises(Exception):
            lbm.Geometry(nx, ny, nz, slab=(z0, z1), porosity=porosity, corr_len=corr_len, seed=seed, **kw)
        return
    want = oracle.geometry(nx, ny, nz, z0, z1, porosity, corr_len, seed)
    g = lbm.Geometry(nx, ny, nz, slab=(z0, z1), porosity=porosity, corr_len=corr_len, seed=seed, **kw)
    assert np.array_equal(g.export()["mask"].reshape(-1), want)
    h = lbm.Geometry(nx, ny, nz, slab=(z0, z1), mask=want.reshape(nz, ny, nx), seed=seed, **kw)
    a, b = g.info(), h.info()
    # (an empty slab of a caller mask means the whole box)
    assert {k: v for k, v in a.items() if z0 < z1 or k != "delta"} == {k: v for k, v in b.items() if z0 < z1 or k != "delta"}
    sim, other = lbm.Simulation(g, p=0.5), lbm.Simulation(h, p=0.5)
    sim.step(2)
    other.set_state(sim.get_state())
