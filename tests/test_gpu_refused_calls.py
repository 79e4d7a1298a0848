"""Calls that CUDA refuses on the host (a reader, which synchronises, on a stream
that is being captured; a step on the capture that this has made void) answer
LBM_ERR_CUDA and leave nothing behind: the calls after them run, with the
results of a simulation that has seen none of it."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_a_refused_call_leaves_no_error_behind():
    import torch
    from paper_1607_02874_gb300 import lbm

    cuda = ctypes.CDLL("libcuda.so.1")
    st = torch.cuda.Stream()
    h = ctypes.c_void_p(st.cuda_stream)
    g = lbm.Geometry(24, 20, 40, slab=(12, 28), porosity=0.6, corr_len=3.0, seed=5, stream=st)
    s, twin = (lbm.Simulation(g, n_species=2, p=0.45, c_init=0.5, stream=st) for _ in "ab")
    out = torch.empty(g.n, device="cuda")
    torch.cuda.synchronize()
    refused = (lambda: s.field_into("rho_C", out), lambda: s.step(1), lambda: lbm.step_batch([s], 1), s.observables,
               s.observables_noalloc)
    after = (lambda x: x.field("rho_R"), lambda x: x.observables()["M_C"], lambda x: x.observables_noalloc()["M_R"],
             lambda x: x.step(2), lambda x: lbm.step_batch([x], 3), lambda x: np.frombuffer(x.get_state(), np.uint8))
    for call in refused:
        for then in after:
            assert cuda.cuStreamBeginCapture_v2(h, 1) == 0  # (mode: thread-local)
            try:
                # the reader makes the capture void, whatever comes second is refused as well
                for c in (refused[0], call):
                    with pytest.raises(lbm.LbmError) as e:
                        c()
                    assert e.value.code == -3
            finally:
                graph = ctypes.c_void_p()
                assert cuda.cuStreamEndCapture(h, ctypes.byref(graph)) != 0 and not graph.value
            a, b = then(s), then(twin)
            if a is not None:
                np.testing.assert_array_equal(a, b)
