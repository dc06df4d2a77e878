"""Profiles where the block sums can go wrong: a bin with more particles than a block may add
up before it flushes, blocks whose range of tiles spans several members of a group.  Counts
are exact; the velocity sums lie within the rounding of the binary64 sums they are compared
with, and a member's profile equals the one it has alone bit for bit."""
import numpy as np
import pytest

import kmc_inputs as ki

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1310_3437_gb300 as kmc  # noqa: E402


def make(n, bins):
    s = ki.piston_setup(n=n, seed=n, profile_bins=bins, profile_every=1)
    return kmc.Simulation(kmc.params_from_setup(s, precision=kmc.KMC_GUARDED_FP32),
                          ki.initial_state(s)), s


@pytest.mark.parametrize("n,bins", [(5001, 256), (300007, 1), (21_000_001, 256), (21_000_001, 3)])
def test_profile_equals_sums_over_the_state(n, bins):
    sim, s = make(n, bins)
    sim.step(1).sync()
    got = sim.profiles()[-1]
    state, _ = sim.state()
    sim.close()
    b = (state[0] * (bins / s.profile_range)).astype(np.int64)
    keep = b < bins
    b = b[keep]
    count = np.bincount(b, minlength=bins)
    assert np.array_equal(got[:, 0], count)
    for k in range(6):
        v = state[3 + k % 3][keep]
        v = v if k < 3 else v * v
        want = np.bincount(b, weights=v, minlength=bins)
        size = np.bincount(b, weights=np.abs(v), minlength=bins)
        # binary64 sum of m terms: m u sum|v|; the digits drop less than 2^-64 a term
        bound = count * (2.0 ** -53 * size * 1.01 + 2.0 ** -64)
        assert np.all(np.abs(got[:, 1 + k] - want) <= bound)


def test_members_of_a_group_equal_themselves_alone():
    sizes = [(70001, 256), (33, 256), (2_600_003, 64), (4097, 7), (300007, 256)]
    alone = [make(n, b)[0] for n, b in sizes]
    members = [make(n, b)[0] for n, b in sizes]
    group = kmc.Group(members)
    for m in members:
        group.budget(m, 2)
    group.step(2)
    group.sync()
    for a, m in zip(alone, members):
        a.step(2).sync()
        pa, pm = a.profiles(), m.profiles()
        assert pa.shape == pm.shape and pa.shape[0] == 2
        assert np.array_equal(pa.view(np.uint64), pm.view(np.uint64))
    group.close()
    for sim in alone + members:
        sim.close()
