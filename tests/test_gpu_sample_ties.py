"""Synthetic samples whose threshold falls among cells of equal value, where the
cell number decides (the lower cell is fluid first): the mask generated on the
device against the oracle's. A box side that equals the smoothing window makes
the field constant along that axis."""
import numpy as np
import pytest

from oracle import oracle

pytestmark = pytest.mark.gpu

CASES = [
    # nx, ny, nz, z0, z1, porosity, corr_len, seed, periodic
    (5, 40, 40, 10, 30, 0.603, 3.0, 5, False),  # rows of 5 equal cells, the threshold after two of one
    (15, 15, 15, 0, 15, 0.5, 10.0, 3, True),  # one value throughout
    (105, 105, 105, 0, 105, 0.41, 74.2, 2, True),  # the same, of more cells than two digits of the cell number hold
]


@pytest.mark.parametrize("nx,ny,nz,z0,z1,porosity,corr_len,seed,periodic", CASES)
def test_ties_go_to_the_lower_cell(nx, ny, nz, z0, z1, porosity, corr_len, seed, periodic):
    from paper_1607_02874_gb300 import lbm

    kw = dict(bc=lbm.BC_PERIODIC) if periodic else {}
    want = oracle.geometry(nx, ny, nz, z0, z1, porosity, corr_len, seed).reshape(nz, ny, nx)
    rows = want[z0:z1].reshape(-1, nx)
    cut = np.flatnonzero(rows.any(1) != rows.all(1))
    assert len(cut) == 1  # the row in which equal cells part
    g = lbm.Geometry(nx, ny, nz, slab=(z0, z1), porosity=porosity, corr_len=corr_len, seed=seed, **kw)
    np.testing.assert_array_equal(g.export()["mask"].reshape(nz, ny, nx), want)
