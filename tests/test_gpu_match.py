"""Matching by pairs where its rounds can go wrong: particles with many candidates (all
four rounds busy, several blocks in the launch of the later rounds), equal keys (a lattice
of counter-moving beams: the partner id decides), and every number of rounds.  Round
counts, partners and state equal the CPU oracle's."""
import numpy as np
import pytest

import kmc_inputs as ki
import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1310_3437_gb300 as kmc  # noqa: E402


def crowded(n):
    """About four candidates per particle: most pairs lose round 0."""
    L = (n / 4096.0) ** (1.0 / 3.0)
    s = ki.equilibrium_setup(n=n, seed=31, L=L, d0=0.09, dt=0.02)
    return s, ki.initial_state(s)


def beams():
    """Particles on a lattice, moving along x in turn by +1 and -1, rows in step: each has
    two partners at the same distance and time of closest approach."""
    m = 12
    g = (np.arange(m) + 0.5) / m
    x, y, z = (a.ravel().copy() for a in np.meshgrid(g, g, g, indexing="ij"))
    sign = np.where(np.arange(m) % 2 == 0, 1.0, -1.0).repeat(m * m)
    s = ki.equilibrium_setup(n=m ** 3, seed=32, d0=0.05, dt=0.06)
    return s, [x, y, z, sign, np.zeros(m ** 3), np.zeros(m ** 3)]


@pytest.mark.parametrize("rounds", [1, 2, 3, 4])
@pytest.mark.parametrize("gas", ["crowded 3000", "crowded 140000", "beams"])
def test_rounds_equal_the_oracle(gas, rounds):
    s, arrays = beams() if gas == "beams" else crowded(int(gas.split()[1]))
    s = s.with_(max_rounds=rounds)
    st = oracle.State(arrays)
    sim = kmc.Simulation(kmc.params_from_setup(s, precision=kmc.KMC_GUARDED_FP32), arrays)
    busy = [0] * 4
    for step in range(2):
        counts, partner, _ = oracle.step(s, st, step)
        sim.step(1).sync()
        got = sim.counts()[-1]
        assert got["edges"] == counts["edges"]
        assert got["round_pairs"] == list(counts["round_pairs"])
        assert np.array_equal(sim.partners(), partner)
        busy = [max(a, b) for a, b in zip(busy, got["round_pairs"])]
    if gas != "beams":
        assert all(b > 0 for b in busy[:rounds]) and not any(busy[rounds:])
    state, last = sim.state()
    for k in range(6):
        assert np.array_equal(state[k].view(np.uint64), st.a[k].view(np.uint64))
    assert np.array_equal(last, st.last)
    sim.close()
