"""The launches of a multi-step call against one-step calls, bit for bit.

Inside one call the wall hits of a step and the next step's emission share a
launch; a call of one step emits before its cell updates and takes its hits
after them, in launches of their own. Both must leave the same state:
populations, observables and checkpoint bytes.
"""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu

BOX = workloads.ragged_case()  # 37 x 29 x 50: partial warps, blocks and node blocks
VARIANTS = {
    "fp32-fluid": dict(layout=2),
    "fp32-dense-det": dict(layout=1, deterministic=True),
    "fp16-fluid-det": dict(layout=2, storage=1, deterministic=True),
    "fp16-cr-fluid": dict(layout=2, storage=1, n_species=1),
    "bf16-random-dense": dict(layout=1, storage=2, sputter=1, sputter_seed=3),
    "fp32-random-fluid-det": dict(layout=2, sputter=1, sputter_seed=4, deterministic=True),
    "fp32-bary": dict(layout=2, velocity=1, c_in=0.05),
    "fp16-bary-random": dict(layout=2, storage=1, velocity=1, c_in=0.05, sputter=1),
    "fp32-channel": dict(layout=2, tau_s=0.6, g_z=1e-5, desorb=True),
    "fp32-bounceback": dict(layout=2, sputter=2),
}


def _state(s):
    o = s.observables(site_map=True)
    return [np.asarray(o[k]) for k in sorted(o)] + [s.populations(), np.frombuffer(s.get_state(), np.uint8)]


def _assert_same(a, b):
    for x, y in zip(_state(a), _state(b)):
        np.testing.assert_array_equal(x, y)


def _sim(lbm, g, **kw):
    return lbm.Simulation(g, **{**dict(n_species=2, p=0.45, pS_P=0.1, c_init=0.5), **kw})


@pytest.mark.parametrize("name", list(VARIANTS))
def test_one_call_equals_single_steps(name):
    from paper_1607_02874_gb300 import lbm

    g = lbm.Geometry(BOX["nx"], BOX["ny"], BOX["nz"], slab=BOX["slab"], porosity=BOX["porosity"],
                     corr_len=BOX["corr_len"], seed=BOX["seed"])
    a, b = _sim(lbm, g, **VARIANTS[name]), _sim(lbm, g, **VARIANTS[name])
    for n in (2, 1, 5, 12):  # calls that start at either parity
        a.step(n)
        for _ in range(n):
            b.step(1)
        _assert_same(a, b)


@pytest.mark.parametrize("n_nodes", [0, 1, 255, 256, 257])
def test_node_counts_around_a_block(n_nodes):
    """Sparse single solid cells: as many catalytic nodes as cells."""
    from paper_1607_02874_gb300 import lbm

    nx, ny, nz = 32, 24, 24
    m = np.zeros((nz, ny, nx), np.uint8)
    at = [(z, y, x) for z in range(3, nz - 3, 2) for y in range(0, ny, 2) for x in range(0, nx, 2)][:n_nodes]
    for c in at:
        m[c] = 1
    g = lbm.Geometry(nx, ny, nz, slab=(2, nz - 2), mask=m)
    assert g.info()["n_nodes"] == n_nodes
    a, b = _sim(lbm, g, storage=1), _sim(lbm, g, storage=1)
    a.step(7)
    for _ in range(7):
        b.step(1)
    _assert_same(a, b)


def test_region_warps_with_and_without_their_own_launch():
    """More region warps than the launch of their own needs (12,288) in one
    box, none in the other: the open planes below the slab evolve alike."""
    from paper_1607_02874_gb300 import lbm

    nx, ny, nz = 128, 128, 64
    out = []
    for fluid in (lbm.LAYOUT_FLUID, lbm.LAYOUT_DENSE):  # dense addressing has no region warps
        g = lbm.Geometry(nx, ny, nz, slab=(52, 60), porosity=0.6, corr_len=4.0, seed=5)
        s = _sim(lbm, g, layout=fluid, p=0.3)
        w = s.warp_counts()
        assert (w["region"] >= 12288) == (fluid == lbm.LAYOUT_FLUID), w
        s.step(9)
        out.append((s.populations(), s.observables(site_map=True)["site_map"]))
    for x, y in zip(*out):
        np.testing.assert_array_equal(x, y)


def test_steps_under_stream_capture():
    """A captured call of two steps, replayed once, leaves what the call leaves."""
    import torch
    from paper_1607_02874_gb300 import lbm

    st = torch.cuda.Stream()
    g = lbm.Geometry(BOX["nx"], BOX["ny"], BOX["nz"], slab=BOX["slab"], porosity=BOX["porosity"],
                     corr_len=BOX["corr_len"], seed=BOX["seed"], stream=st)
    a, b = (_sim(lbm, g, layout=2, storage=1, stream=st) for _ in range(2))
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=st):
        a.step(2)
    with torch.cuda.stream(st):
        graph.replay()
    b.step(2)
    torch.cuda.synchronize()
    _assert_same(a, b)


@pytest.mark.parametrize("side,storage,n_species", [(512, 0, 1), (512, 1, 2), (512, 2, 1), (640, 2, 2), (384, 0, 2)])
def test_wide_planes_against_the_batched_launches(side, storage, n_species):
    """Planes large enough for the odd step's other kernels, which a batch
    never takes; region warps above and below their launch's threshold."""
    from paper_1607_02874_gb300 import lbm

    for nz, slab in ((10, (4, 7)), (16, (9, 13))):
        g = lbm.Geometry(side, side, nz, slab=slab, porosity=0.6, corr_len=4.0, seed=7)
        a, b = (_sim(lbm, g, layout=2, storage=storage, n_species=n_species) for _ in range(2))
        a.step(5)
        lbm.step_batch([b], 5)
        np.testing.assert_array_equal(np.frombuffer(a.get_state(), np.uint8), np.frombuffer(b.get_state(), np.uint8))
