"""A cooperative launch that CUDA refuses, faked on the host by a shim in front of the
runtime's entry point.  Refused once, while the step is captured: the graph without the later
matching rounds is not used, and the steps equal the oracle's.  Refused always: the call fails
with KMC_ECUDA, no step is taken, and the simulation stays failed."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SHIM = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stdlib.h>
struct dim3 { unsigned x, y, z; };
typedef int (*launch_t)(const void*, struct dim3, struct dim3, void**, size_t, void*);
int cudaLaunchCooperativeKernel(const void* f, struct dim3 g, struct dim3 b, void** a, size_t m, void* s) {
  static int left = -1;
  if (left < 0) left = atoi(getenv("REFUSE"));
  if (left > 0) { --left; return 82; }  /* cudaErrorCooperativeLaunchTooLarge */
  return ((launch_t)dlsym(RTLD_NEXT, "cudaLaunchCooperativeKernel"))(f, g, b, a, m, s);
}
"""

CHILD = r"""
import sys
import numpy as np
import kmc_inputs as ki, oracle
import paper_1310_3437_gb300 as kmc

s = ki.equilibrium_setup(n=3000, seed=31, L=(3000 / 4096.0) ** (1.0 / 3.0), d0=0.09, dt=0.02)
arrays = ki.initial_state(s)
def make():
    return kmc.Simulation(kmc.params_from_setup(s, precision=kmc.KMC_GUARDED_FP32), arrays)
sim = make()
members = [make(), make()]
st = oracle.State(arrays)
def same(x, want):
    state, _ = x.state()
    return all(np.array_equal(state[k].view(np.uint64), want[k].view(np.uint64)) for k in range(6))
if sys.argv[1] == "once":
    counts, _ = oracle.run(s, st, 0, 3)
    assert all(min(c["round_pairs"]) > 0 for c in counts)  # the later rounds have work
    sim.step(3).sync()
    assert [c["round_pairs"] for c in sim.counts()] == [list(c["round_pairs"]) for c in counts]
    assert same(sim, st.a)
else:
    group = kmc.Group(members)
    for m in members:
        group.budget(m, 3)
    def code(call):
        try:
            call()
        except kmc.KmcError as e:
            return e.code, "refused" in str(e)
    assert code(lambda: sim.step(3)) == (kmc.KMC_ECUDA, True)
    assert code(sim.sync) == (kmc.KMC_ECUDA, True)
    assert code(lambda: group.step(3))[0] == kmc.KMC_ECUDA
    assert code(group.sync)[0] == kmc.KMC_ECUDA
    for x in [sim] + members:
        assert x.counts() == [] and same(x, arrays)
    group.close()
print("as expected")
"""


@pytest.mark.parametrize("mode,times", [("once", 1), ("always", 1 << 30)])
def test_refused_cooperative_launch(tmp_path, mode, times):
    src, lib = tmp_path / "shim.c", tmp_path / "shim.so"
    src.write_text(SHIM)
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", str(src), "-o", str(lib), "-ldl"], check=True)
    env = dict(os.environ, LD_PRELOAD=str(lib), REFUSE=str(times), PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, "-c", CHILD, mode], cwd=ROOT, env=env, capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0 and "as expected" in r.stdout, r.stderr[-2000:]
