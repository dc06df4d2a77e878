"""The failure path of the matching rounds' barrier.  A test flag keeps it shut: the blocks run
into their bounded wait, the step is abandoned with the timeout status, steps queued behind it
do not wait again, members of a group that do not run the step keep their state, and the device
stays usable."""
import time

import numpy as np
import pytest

import kmc_inputs as ki
import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1310_3437_gb300 as kmc  # noqa: E402


def make(s, arrays, precision, flags=0):
    return kmc.Simulation(kmc.params_from_setup(s, precision=precision, flags=flags), arrays)


def assert_runs(sim, s, arrays, steps):
    st = oracle.State(arrays)
    oracle.run(s, st, 0, steps)
    sim.step(steps).sync()
    state, last = sim.state()
    for k in range(6):
        assert np.array_equal(state[k].view(np.uint64), st.a[k].view(np.uint64))
    assert np.array_equal(last, st.last)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n", [4096, 140000])
def test_timeout_is_reported_once(n, precision):
    s = ki.equilibrium_setup(n=n, seed=71, L=(n / 4096.0) ** (1.0 / 3.0))
    arrays = ki.initial_state(s)
    sim = make(s, arrays, precision, kmc.KMC_FLAG_ROUND_WAIT_TEST)
    t0 = time.perf_counter()
    sim.step(200)
    with pytest.raises(kmc.KmcError) as e:
        sim.sync()
    took = time.perf_counter() - t0
    print(f"one wait: {took:.3f} s")
    assert took < 10.0  # one wait, not one for each queued step
    assert e.value.code == kmc.KMC_ETIMEOUT and "matching rounds" in str(e.value)
    assert sim.counts() == []  # the abandoned step left no record
    state, _ = sim.state()
    for k in range(6):
        assert np.array_equal(state[k], arrays[k])
    sim.close()
    ok = make(s, arrays, precision)
    assert_runs(ok, s, arrays, 3)
    ok.close()


def test_idle_member_of_a_group_keeps_running():
    s = ki.equilibrium_setup(n=3000, seed=72)
    arrays = ki.initial_state(s)
    stuck = make(s, arrays, 1, kmc.KMC_FLAG_ROUND_WAIT_TEST)
    beside, idle = make(s, arrays, 1), make(s, arrays, 1)
    group = kmc.Group([stuck, beside, idle])
    group.budget(stuck, 4)
    group.budget(beside, 4)
    group.step(4)
    with pytest.raises(kmc.KmcError) as e:
        group.sync()
    assert e.value.code == kmc.KMC_ETIMEOUT
    assert stuck.counts() == [] and beside.counts() == []
    group.remove(idle)
    assert_runs(idle, s, arrays, 3)
    group.close()
    for sim in (stuck, beside, idle):
        sim.close()
