"""Per-step batched launches against the same simulations alone, bit for bit:
runs of either parity, groups with and without a launch of their own for the
region warps, and a group whose species bounce back in some members."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _state(s):
    return [s.populations(), np.frombuffer(s.get_state(), np.uint8)]


def _compare(lbm, make, ages, steps):
    """make(k): simulation k twice over; ages[k]: the steps it has behind it."""
    pairs = [make(k) for k in range(len(ages))]
    for (a, b), n in zip(pairs, ages):
        if n:
            a.step(n)
            b.step(n)
    for n in steps:
        lbm.step_batch([a for a, _ in pairs], n)
        for a, b in pairs:
            b.step(n)
            for x, y in zip(_state(a), _state(b)):
                np.testing.assert_array_equal(x, y)


@pytest.mark.parametrize("layout", ["fluid", "dense"])
@pytest.mark.parametrize("ages", [(0, 0, 0), (1, 1), (0, 1, 0, 3), (1,), (2, 1) * 8], ids=str)
def test_runs_of_either_parity(ages, layout):
    from paper_1607_02874_gb300 import lbm

    code = lbm.LAYOUT_FLUID if layout == "fluid" else lbm.LAYOUT_DENSE

    def make(k):
        g = lbm.Geometry(17 + k, 13, 24, slab=(6, 18), porosity=0.6, corr_len=2.0, seed=40 + k)
        return [lbm.Simulation(g, n_species=2, p=0.4, pS_P=0.1, c_init=0.5, storage=lbm.FP16_DEV, layout=code) for _ in "ab"]

    _compare(lbm, make, ages, (1, 4))


@pytest.mark.parametrize("storage", ["FP32", "FP16_DEV"])
@pytest.mark.parametrize("n_species", [1, 2])
def test_region_warps_of_a_batch(storage, n_species):
    """Two boxes that together hold the 12,288 region warps, one that holds
    none, at both parities."""
    from paper_1607_02874_gb300 import lbm

    def make(k):
        n = (128, 128, 24, (17, 20)) if k < 2 else (20, 18, 16, (3, 13))
        g = lbm.Geometry(*n[:3], slab=n[3], porosity=0.6, corr_len=3.0, seed=60 + k)
        return [lbm.Simulation(g, n_species=n_species, p=0.4, c_init=0.5, storage=getattr(lbm, storage),
                               layout=lbm.LAYOUT_FLUID) for _ in "ab"]

    pair = [make(k)[0].warp_counts()["region"] for k in range(3)]
    assert pair[0] < 12288 <= pair[0] + pair[1] and pair[2] == 0, pair
    _compare(lbm, make, (0, 1, 1), (3, 2))


def test_species_bounce_back_beside_catalytic_members():
    from paper_1607_02874_gb300 import lbm

    def make(k):
        g = lbm.Geometry(22, 15, 26, slab=(7, 19), porosity=0.6, corr_len=2.0, seed=80 + k)
        kw = dict(sputter=2) if k % 2 else dict(tau_s=0.6)
        return [lbm.Simulation(g, n_species=2, p=0.4, c_init=0.5, **kw) for _ in "ab"]

    _compare(lbm, make, (0, 0, 1, 1), (1, 6))
