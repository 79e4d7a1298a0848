"""The state readers against one another: a field's kernel reads the carrier's
populations, the species' or both; all of them must say what the exported
populations (which read everything) say, in both parities, and so must the
plane sums, with the two observable calls equal to the bit."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu

R = workloads.ragged_case()
BOXES = {
    "ragged": (R["nx"], R["ny"], R["nz"], R["slab"]),  # partial warps, blocks and shares of a plane
    "column": (1, 1, 8, (3, 5)),                        # planes of one cell
    "wide": (67, 61, 9, (3, 6)),                        # planes of more cells than a cluster has threads
}
MODES = {
    "fp32": dict(),
    "fp32-cr-dense": dict(n_species=1, layout=1),
    "fp16-det": dict(storage=1, deterministic=True),
    "bf16-random-dense": dict(storage=2, sputter=1, layout=1),
    "fp32-bary": dict(velocity=1, c_in=0.05),
    "fp32-force": dict(g_z=1e-5, tau_s=0.6),
    "fp16-bounceback": dict(storage=1, sputter=2),
}
CX = np.array([0, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, 1, -1, 0, 0, 0, 0])
CY = np.array([0, 0, 0, 1, -1, 0, 0, 1, -1, -1, 1, 0, 0, 0, 0, 1, -1, 1, -1])
CZ = np.array([0, 0, 0, 0, 0, 1, -1, 0, 0, 0, 0, 1, -1, -1, 1, 1, -1, -1, 1])


@pytest.mark.parametrize("mode", list(MODES))
@pytest.mark.parametrize("box", list(BOXES))
def test_fields_and_sums_follow_from_the_populations(box, mode):
    from paper_1607_02874_gb300 import lbm

    nx, ny, nz, slab = BOXES[box]
    g = lbm.Geometry(nx, ny, nz, slab=slab, porosity=0.6, corr_len=3.0, seed=7)
    kw = {**dict(n_species=2, p=0.45, pS_P=0.1, c_init=0.5, layout=2), **MODES[mode]}
    s = lbm.Simulation(g, **kw)
    inside = np.zeros((nz, ny * nx), bool)
    inside[1:-1] = True
    inside = inside.reshape(-1) & (g.export()["mask"] == 0)
    for n in (6, 1):  # an even state, then an odd one
        s.step(n)
        f = s.populations().astype(np.float64)
        size = np.abs(f).sum(1)  # a sum of 19 rounded terms is within 19 units of 2^-24 of this
        rho, j = f.sum(1), [(c[None, :, None] * f).sum(1) for c in (CX, CY, CZ)]
        bary = kw.get("velocity") == 1
        over = 1.0 + (rho.sum(0) if bary else rho[0])
        want = {"drho_C": rho[0], "rho_R": rho[1], "rho_C": 1.0 + rho[0]}
        tol = {"drho_C": 19 * 2.0 ** -24 * size[0], "rho_R": 19 * 2.0 ** -24 * size[1],
               "rho_C": 20 * 2.0 ** -24 * (1.0 + size[0])}
        if kw["n_species"] == 2:
            want["rho_P"], tol["rho_P"] = rho[2], 19 * 2.0 ** -24 * size[2]
        for k, name in enumerate(("ux", "uy", "uz")):
            want[name] = (j[k].sum(0) if bary else j[k][0]) / over + (0.5 * kw.get("g_z", 0.0) if name == "uz" else 0.0)
            tol[name] = 60 * 2.0 ** -24 * (size.sum(0) if bary else size[0]) + 2.0 ** -23 * (np.abs(want[name]) + 1e-9)
        got = {}
        for name, w in want.items():
            got[name] = s.field(name).astype(np.float64)
            assert not got[name][~inside].any(), name
            d = np.abs(got[name] - w)[inside]
            assert (d <= tol[name][inside]).all(), (name, d.max())
        o, q = s.observables(), s.observables_noalloc(profiles=True)
        for k in q:
            np.testing.assert_array_equal(q[k], o[k], err_msg=k)
        # the plane sums round each cell's moments in an order of their own:
        # every cell within the bound of its field
        plane = lambda v: np.where(inside, v, 0.0).reshape(nz, -1).sum(1)  # noqa: E731
        sums = {"rhoC_z": (want["rho_C"], tol["rho_C"]), "rhoR_z": (want["rho_R"], tol["rho_R"])}
        if kw["n_species"] == 2:
            P, u = want["rho_P"], want["uz"]
            sums["rhoP_z"] = (P, tol["rho_P"])
            sums["phiP_z"] = (P * u, np.abs(P) * tol["uz"] + (np.abs(u) + tol["uz"]) * tol["rho_P"])
        for k, (w, t) in sums.items():
            assert (np.abs(o[k] - plane(w)) <= plane(t) + 1e-12 * plane(np.abs(w))).all(), k
