"""A launch that fails in the middle of a call, made on the host: a stand-in for
the step's launch functions hands one error back to the library in place of a
launch. The call reports it, every simulation stands at the steps it has run,
its observables are those of that step, and stepping on gives what an
undisturbed simulation gives, bit for bit.

Runs in a child process, which loads the stand-in ahead of the library so that
the library's own calls find it. No kernel is made to fault, trap or hang."""
import os
import subprocess
import sys
import textwrap

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# launch_step_st and launch_batch_split_st of the FP32 carrier variant: count
# down, return cudaErrorMemoryAllocation (2) once, else pass on to the library's
STAND_IN = r"""
#include <dlfcn.h>
enum cudaError : unsigned { kOk = 0, kNoMemory = 2 };
struct CUstream_st;
struct CUevent_st;
static void *lib;
static long left = -1;
extern "C" void stand_in(const char *path, long n) {
  if (!lib) lib = dlopen(path, RTLD_NOLOAD | RTLD_NOW);
  left = n;
}
static bool fails() { return left >= 0 && left-- == 0; }
namespace lbm {
struct StepArgs;
struct BatchLaunch;
template <int ST, bool RS, int PHYS>
cudaError launch_step_st(const StepArgs &a, int layout, int ns, int parity, CUstream_st *st, CUevent_st *const *ev,
                         bool first, bool last) {
  using F = cudaError (*)(const StepArgs &, int, int, int, CUstream_st *, CUevent_st *const *, bool, bool);
  if (fails()) return kNoMemory;
  return ((F)dlsym(lib, "STEP"))(a, layout, ns, parity, st, ev, first, last);
}
template <int ST, bool RS, int PHYS>
cudaError launch_batch_split_st(const BatchLaunch &p, int layout, int ns, int det, CUstream_st *st, bool first, bool last) {
  using F = cudaError (*)(const BatchLaunch &, int, int, int, CUstream_st *, bool, bool);
  if (fails()) return kNoMemory;
  return ((F)dlsym(lib, "BATCH"))(p, layout, ns, det, st, first, last);
}
template cudaError launch_step_st<0, false, 0>(const StepArgs &, int, int, int, CUstream_st *, CUevent_st *const *, bool, bool);
template cudaError launch_batch_split_st<0, false, 0>(const BatchLaunch &, int, int, int, CUstream_st *, bool, bool);
}
"""

CHILD = r"""
import ctypes, sys
import numpy as np
so, deterministic = sys.argv[1], sys.argv[2] == "det"
fake = ctypes.CDLL(so, mode=ctypes.RTLD_GLOBAL)
from paper_1607_02874_gb300 import lbm
from paper_1607_02874_gb300.build import LIB
lbm.library()

def fail_at(n):
    fake.stand_in(LIB.encode(), ctypes.c_long(n))

def geometry(seed):
    return lbm.Geometry(24, 20, 40, slab=(12, 28), porosity=0.6, corr_len=3.0, seed=seed)

G = [geometry(k) for k in range(3)]

def sim(k, **kw):
    return lbm.Simulation(G[k], **{**dict(n_species=2, p=0.45, pS_P=0.1, c_init=0.5, layout=lbm.LAYOUT_FLUID,
                                          deterministic=deterministic), **kw})

def same(a, b, whole):
    x, y = a.observables(site_map=True), b.observables(site_map=True)
    for k in sorted(y):
        np.testing.assert_array_equal(np.asarray(x[k]), np.asarray(y[k]), err_msg=k)
    x, y = a.observables_noalloc(), b.observables_noalloc()
    assert x == y, (x, y)
    np.testing.assert_array_equal(a.populations(), b.populations())
    if whole:
        assert a.get_state() == b.get_state()

def refused(call):
    try:
        call()
    except lbm.LbmError as e:
        assert e.code == -3, e
        return
    raise AssertionError("the failed launch was not reported")

fail_at(-1)
for start in (0, 3):
    for k in (0, 1, 4):  # the launch of step k of six fails
        a, b = sim(0), sim(0)
        if start:
            a.step(start); b.step(start)
        fail_at(k)
        refused(lambda: a.step(6))
        fail_at(-1)
        assert a.info()["step"] == start + k
        if k:
            b.step(k)
        same(a, b, False)
        a.step(6 - k); b.step(6 - k)
        same(a, b, True)

# a batch of two groups (one species, two species): the first group of a
# batch's step runs, the second one's launch fails
for k in (1, 2, 7):
    kws = [(0, dict(n_species=1)), (1, dict()), (2, dict(n_species=1))]
    sims, twins = [sim(q, **kw) for q, kw in kws], [sim(q, **kw) for q, kw in kws]
    sims[2].step(1); twins[2].step(1)
    fail_at(k)
    refused(lambda: lbm.step_batch(sims, 6))
    fail_at(-1)
    ran = [(k + 1) // 2, k // 2, (k + 1) // 2]
    for s, t, r, past in zip(sims, twins, ran, (0, 0, 1)):
        assert s.info()["step"] == past + r, (k, s.info())
        if r:
            t.step(r)
        same(s, t, False)
        s.step(5); t.step(5)
        same(s, t, True)
print("as undisturbed")
"""


def _mangled(lib, name):
    out = subprocess.run(["nm", "-D", "--defined-only", lib], capture_output=True, text=True, check=True).stdout
    found = [w for w in out.split() if name in w]
    assert len(found) == 1, (name, found)
    return found[0]


@pytest.mark.parametrize("hits", ["fp32", "det"])
def test_a_failed_launch_leaves_the_steps_before_it(tmp_path, hits):
    from paper_1607_02874_gb300.build import LIB

    src = STAND_IN.replace('"STEP"', '"%s"' % _mangled(LIB, "launch_step_stILi0ELb0ELi0E"))
    src = src.replace('"BATCH"', '"%s"' % _mangled(LIB, "launch_batch_split_stILi0ELb0ELi0E"))
    cc, so = tmp_path / "stand_in.cpp", tmp_path / "stand_in.so"
    cc.write_text(src)
    subprocess.run(["g++", "-shared", "-fPIC", "-O1", "-o", str(so), str(cc), "-ldl"], check=True)
    r = subprocess.run([sys.executable, "-c", textwrap.dedent(CHILD), str(so), hits], cwd=ROOT,
                       env=dict(os.environ, PYTHONPATH=ROOT), capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and "as undisturbed" in r.stdout, r.stdout[-2000:] + r.stderr[-4000:]
