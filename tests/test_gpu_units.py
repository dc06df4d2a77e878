"""Lengths in any unit.  A gas and its copies with every length, and either dt or every
velocity, times a power of two are the same gas to the last bit: pair lists, partners and state
of the copies equal those of the original, which equal the CPU oracle's.  The pair filter of
the tiled search works in squares of lengths; beyond what its operands hold it passes every
pair (2^-100 and 2^95 below), as in a gas in one cell much smaller than d0."""
import numpy as np
import pytest

import kmc_inputs as ki
import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1310_3437_gb300 as kmc  # noqa: E402

UNITS = [-100, -75, -70, -62, -40, 40, 62, 70, 80, 95]


def gas(kind):
    s = ki.equilibrium_setup(n=3000, seed=21, d0=0.03, dt=0.004)
    if kind == "dense":  # about 30 particles per cell
        s = s.with_(dt=0.012)
    if kind == "walls":
        s = s.with_(box=(0.5, 1.0, 1.0), bc=(ki.REFLECT, ki.REFLECT, ki.PERIODIC),
                    piston_x0=0.5, piston_u=0.25)
    rng = np.random.default_rng(21)
    return s, [rng.random(s.n) * b for b in s.box] + [rng.standard_normal(s.n) for _ in range(3)]


def scaled(s, arrays, length, speed):
    """Lengths times 2^length, velocities times 2^speed, dt to match."""
    f, v = 2.0 ** length, 2.0 ** speed
    s = s.with_(box=tuple(b * f for b in s.box), d0=s.d0 * f, dt=s.dt * f / v,
                piston_x0=s.piston_x0 * f, piston_u=s.piston_u * v)
    return s, [a * f for a in arrays[:3]] + [a * v for a in arrays[3:]]


def compare(s, arrays, units, precision, kernel, flags, steps=3):
    """units: (length, speed) exponents"""
    st = oracle.State(arrays)
    sims = [kmc.Simulation(kmc.params_from_setup(c[0], precision=precision, search_kernel=kernel,
                                                 flags=flags), c[1])
            for c in (scaled(s, arrays, *u) for u in units)]
    found = 0
    for step in range(steps):
        pi, pj, _, _ = oracle.candidate_pairs(s, st)
        _, partner, _ = oracle.step(s, st, step)
        want = np.stack([pi, pj], axis=1)
        found += len(want)
        for u, sim in zip(units, sims):
            sim.step(1).sync()
            assert np.array_equal(sim.edges(), want), (u, step)
            assert np.array_equal(sim.partners(), partner), (u, step)
    assert found > 0
    for (length, speed), sim in zip(units, sims):
        state, last = sim.state()
        for k in range(6):
            back = state[k] * 2.0 ** -(length if k < 3 else speed)
            assert np.array_equal(back.view(np.uint64), st.a[k].view(np.uint64)), (length, speed)
        assert np.array_equal(last, st.last)
        sim.close()


@pytest.mark.parametrize("kernel", [0, 1])
@pytest.mark.parametrize("kind", ["box", "dense", "walls"])
def test_binary64_in_any_unit(kind, kernel):
    """without the speed split (flags 1): every pair is a slow one"""
    units = [(0, 0), (40, -100)] + [(u, 0) for u in UNITS] + [(u, u) for u in UNITS if -75 <= u <= 40]
    compare(*gas(kind), units, kmc.KMC_FP64, kernel, flags=1)


@pytest.mark.parametrize("kernel", [0, 1])
@pytest.mark.parametrize("kind", ["box", "walls"])
def test_binary64_split_in_any_unit(kind, kernel):
    """with the speed split whenever it fits (flags 2): the fast particles' reach, too"""
    units = [(0, 0), (40, -100)] + [(u, 0) for u in UNITS] + [(u, u) for u in UNITS if -75 <= u <= 40]
    s, arrays = gas(kind)
    compare(s.with_(d0=0.015, dt=0.002), arrays, units, kmc.KMC_FP64, kernel, flags=2)


@pytest.mark.parametrize("flags", [0, 1])
@pytest.mark.parametrize("kind", ["box", "dense", "walls"])
def test_binary32_tiles_in_common_units(kind, flags):
    """nanometres to kilometres, picoseconds to seconds"""
    units = [(u, v) for u in (-30, -10, 0, 10) for v in (-10, 0, 10)]
    compare(*gas(kind), units, kmc.KMC_GUARDED_FP32, 2, flags)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("d0", [0.7, 1.2, 1.6, 3.0, 40.0, 1e3, 1e6])
def test_one_cell_smaller_than_d0(d0, precision):
    """the threshold of the filter grows as (d0 / box)^2"""
    rng = np.random.default_rng(5)
    s = ki.equilibrium_setup(n=90, seed=5, d0=d0, dt=0.05).with_(
        bc=(ki.REFLECT,) * 3, piston_x0=1.0)
    arrays = [rng.random(s.n) for _ in range(3)] + [rng.standard_normal(s.n) for _ in range(3)]
    compare(s, arrays, [(0, 0), (-70, 0), (70, 0)] if precision == 0 else [(0, 0)], precision, 2, 1)
