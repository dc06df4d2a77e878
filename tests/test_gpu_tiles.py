"""The tiled search (search_kernel 2, and every binary64 step) where its tiles have edges:
partial rows and partner tiles, short periodic axes whose ranges wrap, columns longer than a
run, cells with many tiles, one-cell axes, the plane.  Pair lists, partners and state equal
the CPU oracle's bit for bit.  The rounding of the pair filter is checked on the CPU."""
import numpy as np
import pytest

import kmc_inputs as ki
import oracle

# name, setup: n just below and above a tile of 32; nx = 3 and 4 cells on a periodic x axis;
# a sparse tube whose runs of 32 span more than 64 cells; about 90 particles per cell; a
# reflecting slab of one cell along z and one along x; particles in the plane
CASES = {
    "one": ki.equilibrium_setup(n=1, seed=1),
    "n31": ki.equilibrium_setup(n=31, seed=2, d0=0.1),
    "n33": ki.equilibrium_setup(n=33, seed=3, d0=0.1),
    "n1025": ki.equilibrium_setup(n=1025, seed=4, d0=0.04),
    "short_x3": ki.equilibrium_setup(n=900, seed=5, d0=0.03, dt=0.004).with_(box=(0.24, 1.0, 1.0)),
    "short_x4": ki.equilibrium_setup(n=900, seed=6, d0=0.03, dt=0.004).with_(box=(0.3, 1.0, 1.0)),
    "sparse_tube": ki.piston_setup(n=500, seed=7, box=(60.0, 0.3, 0.3), profile_bins=0,
                                   profile_every=0).with_(d0=0.02, dt=0.005),
    "dense": ki.equilibrium_setup(n=6000, seed=8, d0=0.02, dt=0.024),
    "slab_z": ki.equilibrium_setup(n=1500, seed=9, d0=0.03, dt=0.004).with_(
        box=(1.0, 1.0, 0.1), bc=(ki.PERIODIC, ki.PERIODIC, ki.REFLECT)),
    "slab_x": ki.equilibrium_setup(n=1500, seed=10, d0=0.03, dt=0.004).with_(
        box=(0.1, 1.0, 1.0), bc=(ki.REFLECT, ki.PERIODIC, ki.REFLECT), piston_x0=0.1),
    "plane": ki.equal_speed_setup(n=3000, seed=11, d0=0.004, dt=0.01),
}


def arrays_of(s):
    if s.name.startswith("equal_speed") or s.name.startswith("piston"):
        return ki.initial_state(s)
    rng = np.random.default_rng(s.seed)
    pos = [np.minimum(rng.random(s.n) * b, np.nextafter(b, 0.0)) for b in s.box]
    return pos + [rng.standard_normal(s.n) for _ in range(3)]


@pytest.mark.gpu
@pytest.mark.parametrize("stencil", [1, 2])
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("name", sorted(CASES))
def test_tiles_equal_the_oracle(name, precision, stencil):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_1310_3437_gb300 as kmc

    s = CASES[name]
    arrays = arrays_of(s)
    st = oracle.State(arrays)
    # flags 1: no speed split, so that every pair is a slow one; the default splits
    sims = [kmc.Simulation(kmc.params_from_setup(s, precision=precision, stencil=stencil,
                                                 search_kernel=2, flags=f), arrays) for f in (1, 0)]
    for step in range(4):
        pi, pj, _, _ = oracle.candidate_pairs(s, st)
        _, partner, _ = oracle.step(s, st, step)
        want = np.stack([pi, pj], axis=1)
        for sim in sims:
            sim.step(1).sync()
            got = sim.edges()
            assert got.shape == want.shape and np.array_equal(got, want), f"step {step}"
            assert np.array_equal(sim.partners(), partner), f"step {step}"
    for sim in sims:
        state, last = sim.state()
        for k in range(6):
            assert np.array_equal(state[k].view(np.uint64), st.a[k].view(np.uint64))
        assert np.array_equal(last, st.last)
        sim.close()


def split16(x):
    hi = x.astype(np.float16)
    return hi.astype(np.float64), (x - hi.astype(np.float32)).astype(np.float16).astype(np.float64)


@pytest.mark.parametrize("extent", [1.0, 0.3, 0.02])
def test_pair_filter_rounding(extent):
    """The operands of the filter represent the form within 2^-14 less the 384 u of the
    inner product's sums (u = 2^-24), and rounding b to binary16 moves |b_i - b_j|^2 by at
    most 2^-7 of the largest |b|^2."""
    rng = np.random.default_rng(0)
    m = 200_000
    a = [(rng.random((2, m)) * 2 - 1).astype(np.float32) * np.float32(extent) for _ in range(3)]
    b = [(rng.random((2, m)) * 2 - 1).astype(np.float32) / np.float32(np.sqrt(3)) for _ in range(3)]
    br = [x.astype(np.float16).astype(np.float32) for x in b]
    s = ((a[0] * a[0] + (a[1] * a[1] + a[2] * a[2])) - (br[0] * br[0] + (br[1] * br[1] + br[2] * br[2])))
    form = sum(sum(split16(s[k])) for k in (0, 1))
    for x in a:
        (hi, lo), (hj, lj) = split16(x[0]), split16(x[1])
        form = form - 2.0 * (hi * hj + hi * lj + lo * hj)
    for x in br:
        form = form + 2.0 * x[0].astype(np.float64) * x[1]
    want = sum((x[0].astype(np.float64) - x[1]) ** 2 for x in a) - \
        sum((x[0].astype(np.float64) - x[1]) ** 2 for x in br)
    assert np.abs(form - want).max() <= (1024 - 384) * 2.0 ** -24
    moved = sum((x[0].astype(np.float64) - x[1]) ** 2 for x in b) - \
        sum((x[0].astype(np.float64) - x[1]) ** 2 for x in br)
    top = sum(x.astype(np.float64) ** 2 for x in b).max()
    assert np.abs(moved).max() <= 2.0 ** -7 * top
