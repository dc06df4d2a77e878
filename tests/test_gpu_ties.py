"""Matching where every choice is a tie: combs of counter-moving particles in which each one
has two partners at bit-equal distance and time of closest approach, on either side of it,
so that only the partner's id decides, and each place is contested by two pairs.  The ids
are shuffled, and the pairs compete from many blocks.  Round counts, partners and state equal
the CPU oracle's."""
import numpy as np
import pytest

import kmc_inputs as ki
import oracle


def combs(seed):
    """Along y (periodic) particles 1/32 apart move by +1 and -1 along x in turn, those moving
    back 1/32 ahead in x: all coordinates are exact, so are all differences.  Layers along z
    and combs along x are too far apart to meet within the step."""
    y, z, x = (a.ravel() for a in np.meshgrid(np.arange(32), np.arange(16), np.arange(8), indexing="ij"))
    back = y % 2 == 1
    pos = [x / 8.0 + back / 32.0, y / 32.0, z / 16.0]
    vx = np.where(back, -1.0, 1.0)
    order = np.random.default_rng(seed).permutation(x.size)
    arrays = [np.ascontiguousarray(a[order]) for a in pos + [vx, 0.0 * vx, 0.0 * vx]]
    return ki.equilibrium_setup(n=x.size, seed=seed, d0=1.5 / 32, dt=0.03), arrays


def test_every_choice_is_a_tie():
    s, arrays = combs(1)
    pi, pj, d2, t = oracle.candidate_pairs(s, oracle.State(arrays))
    ends = np.concatenate([pi, pj])
    assert np.array_equal(np.bincount(ends, minlength=s.n), np.full(s.n, 2))
    assert np.unique(d2).size == 1 and np.unique(t).size == 1


@pytest.mark.gpu
@pytest.mark.parametrize("rounds", [1, 2, 3, 4])
@pytest.mark.parametrize("precision,kernel", [(0, 1), (1, 3)])
def test_ties_equal_the_oracle(precision, kernel, rounds):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_1310_3437_gb300 as kmc

    for seed in range(4):
        s, arrays = combs(seed)
        s = s.with_(max_rounds=rounds)
        st = oracle.State(arrays)
        sim = kmc.Simulation(kmc.params_from_setup(s, precision=precision, search_kernel=kernel), arrays)
        counts, partner, _ = oracle.step(s, st, 0)
        sim.step(1).sync()
        got = sim.counts()[-1]
        assert got["edges"] == counts["edges"] == s.n
        assert got["round_pairs"] == list(counts["round_pairs"])
        assert min(got["round_pairs"][:rounds]) > 0
        assert np.array_equal(sim.partners(), partner)
        state, last = sim.state()
        for k in range(6):
            assert np.array_equal(state[k].view(np.uint64), st.a[k].view(np.uint64))
        assert np.array_equal(last, st.last)
        sim.close()
