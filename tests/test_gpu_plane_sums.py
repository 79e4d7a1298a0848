"""Plane sums where the number of blocks that share a plane changes (eight, four,
two or one, by the planes' size and number), and where the allocation-free
observables' planes fill one tile, more than one, or part of the last: both
observable calls equal to the bit, and their profiles what the exported
populations say."""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

BOXES = [
    # nx, ny, nz, periodic: on either side of each line
    (32, 32, 38, False), (32, 32, 39, False), (45, 45, 39, False), (46, 46, 39, False),
    (77, 80, 39, False), (77, 79, 40, True), (80, 80, 114, False), (80, 80, 115, False),
    (16, 16, 76, False), (16, 16, 77, True), (16, 16, 152, False), (16, 16, 153, False),
    (6, 5, 256, False), (6, 5, 257, False), (6, 5, 600, True),
]


def _box(lbm, nx, ny, nz, periodic, **kw):
    mid = min(nz // 2, 256)
    g = lbm.Geometry(nx, ny, nz, slab=(max(3, mid - nz // 4), mid + nz // 4), porosity=0.6, corr_len=2.0, seed=9,
                     **(dict(bc=lbm.BC_PERIODIC) if periodic else {}))
    return g, lbm.Simulation(g, **{**dict(n_species=2, p=0.45, pS_P=0.1, c_init=0.5, rho_in=1.0), **kw})


@pytest.mark.parametrize("nx,ny,nz,periodic", BOXES)
@pytest.mark.parametrize("storage,layout", [("FP32", 2), ("FP16_DEV", 1)])
def test_profiles_follow_from_the_populations(nx, ny, nz, periodic, storage, layout):
    from paper_1607_02874_gb300 import lbm

    g, s = _box(lbm, nx, ny, nz, periodic, storage=getattr(lbm, storage), layout=layout)
    inside = g.export()["mask"].reshape(nz, -1) == 0
    if not periodic:
        inside[[0, -1]] = False
    for n in (4, 1):  # an even state, then an odd one
        s.step(n)
        o, q = s.observables(site_map=True), s.observables_noalloc(profiles=True)
        for k in q:
            np.testing.assert_array_equal(q[k], o[k], err_msg=k)
        f = s.populations().reshape(3, 19, nz, -1).astype(np.float64)
        size = np.abs(f).sum(1)  # a sum of 19 rounded terms is within 19 units of 2^-24 of this
        for k, name in enumerate(("rhoC_z", "rhoR_z", "rhoP_z")):
            rho = np.where(inside, f[k].sum(0) + (k == 0), 0.0).sum(1)
            tol = np.where(inside, 20 * 2.0 ** -24 * (size[k] + (k == 0)), 0.0).sum(1)
            assert (np.abs(o[name] - rho) <= tol + 1e-12 * np.abs(rho)).all(), name
        # (each node's share is one FP32 product)
        assert o["react_z"].sum() == pytest.approx(o["site_map"].astype(np.float64).sum(), rel=1e-6)
        assert o["site_map"].any()


@pytest.mark.parametrize("nx,ny,nz", [(46, 46, 912), (46, 46, 913), (128, 128, 228), (128, 128, 229)])
@pytest.mark.parametrize("layout", [1, 2])
def test_profiles_follow_from_the_fields(nx, ny, nz, layout):
    from paper_1607_02874_gb300 import lbm

    g, s = _box(lbm, nx, ny, nz, False, layout=layout)
    s.step(3)
    o, q = s.observables(), s.observables_noalloc(profiles=True)
    for k in q:
        np.testing.assert_array_equal(q[k], o[k], err_msg=k)
    for name in ("rho_C", "rho_R"):  # (both sides round 19 terms of a cell: 2 x 19 units of 2^-24)
        want = s.field(name).reshape(nz, -1)[1:-1].astype(np.float64).sum(1)
        np.testing.assert_allclose(o[name.replace("_", "") + "_z"][1:-1], want, rtol=1e-5)


def test_many_small_planes_are_read_fast():
    """Planes of 256 cells cost 0.08 us each with one block to a plane; eight
    blocks to each took 0.3."""
    from paper_1607_02874_gb300 import lbm

    nz = 4000
    g, s = _box(lbm, 16, 16, nz, False)
    took = []
    for _ in range(30):
        t = time.perf_counter()
        s.observables_noalloc()
        took.append(time.perf_counter() - t)
    assert min(took) < 0.2e-6 * nz, min(took)
