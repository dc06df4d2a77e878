"""Particles outside the box: a reflecting wall acts once a step, so a particle that crosses a
thin slab more than once within a step ends it beyond a wall, and a simulation may start with
particles beyond a piston that has already moved.  The binary64 searches find the oracle's
pairs (all pairs tested) all the same, alone and decomposed."""
import numpy as np
import pytest

import kmc_inputs as ki
import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1310_3437_gb300 as kmc  # noqa: E402


def check(s, arrays, steps, step0=0, domains=None, outside=True, flags=1, kernel=2):
    p = kmc.params_from_setup(s, precision=kmc.KMC_FP64, search_kernel=kernel, flags=flags, step0=step0,
                              edge_cap=1 << 16)
    sim = kmc.Simulation(p, arrays) if domains is None else kmc.Simulation(p, arrays, domains=domains)
    st = oracle.State(arrays)
    far = 0.0
    for step in range(step0, step0 + steps):
        pi, pj, _, _ = oracle.candidate_pairs(s, st, search=0)
        _, partner, _ = oracle.step(s, st, step, search=0)
        sim.step(1).sync()
        assert np.array_equal(sim.edges(), np.stack([pi, pj], axis=1)), step
        assert np.array_equal(sim.partners(), partner), step
        far = max([far] + [float(max(-st.a[k].min(), st.a[k].max() - s.box[k])) for k in range(3)])
    assert outside is None or (far > 0.0) == outside
    state, _ = sim.state()
    for k in range(6):
        assert np.array_equal(state[k].view(np.uint64), st.a[k].view(np.uint64))
    sim.close()


def gas(n, box, bc, seed, d0, dt, **kw):
    s = ki.equilibrium_setup(n=n, seed=seed, d0=d0, dt=dt).with_(box=box, bc=bc, piston_x0=box[0], **kw)
    rng = np.random.default_rng(seed)
    return s, [rng.random(n) * b for b in box] + [rng.standard_normal(n) for _ in range(3)]


@pytest.mark.parametrize("kernel", [0, 1])
@pytest.mark.parametrize("thin", [0.02, 0.004, 1e-4])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_thin_slab(axis, thin, kernel):
    box, bc = [1.0, 1.0, 1.0], [ki.PERIODIC] * 3
    box[axis], bc[axis] = thin, ki.REFLECT
    check(*gas(2500, tuple(box), tuple(bc), 41 + axis, 0.02, 0.02), 6, kernel=kernel)


@pytest.mark.parametrize("domains", [1, 2])
def test_thin_slab_decomposed(domains):
    check(*gas(2500, (1.0, 1.0, 0.004), (ki.PERIODIC, ki.PERIODIC, ki.REFLECT), 44, 0.02, 0.02), 5,
          domains=domains)


@pytest.mark.parametrize("step0", [40, 95, 99])
def test_beyond_the_piston(step0):
    """The wall stands at 1 - step0 / 100 of the box."""
    s, arrays = gas(2500, (1.0, 1.0, 1.0), (ki.REFLECT,) * 3, 45, 0.02, 0.004, piston_u=2.5)
    check(s, arrays, 1, step0=step0, outside=None)


def test_inside():
    """in a box that no particle crosses, the same calls take the filtered search"""
    check(*gas(2500, (1.0, 1.0, 0.2), (ki.PERIODIC, ki.PERIODIC, ki.REFLECT), 46, 0.02, 0.02), 4,
          outside=False)
