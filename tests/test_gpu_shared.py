"""Small simulations, whose searches share the partners of 32 particles among two, four or
eight warps, against the same simulations as members of a group too large for that (a warp
each): state, partners and every count of every step are equal.  Sizes at the edges of a
warp, of a block and of the three ways to share; both searches, periodic and bounded x axis,
with and without the speed split."""
import numpy as np
import pytest

import kmc_inputs as ki

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1310_3437_gb300 as kmc  # noqa: E402

SIZES = [1, 33, 257, 4097, 19457, 38913, 77825]


def setup_of(n, gas):
    if gas == "tube":
        s = ki.piston_setup(n=n, seed=n, profile_bins=0, profile_every=0)
    else:
        s = ki.equilibrium_setup(n=n, seed=n, L=(n / 4096.0) ** (1.0 / 3.0))
    return s, ki.initial_state(s)


@pytest.mark.parametrize("stencil", [1, 2])
@pytest.mark.parametrize("gas", ["box", "tube"])
@pytest.mark.parametrize("search", ["rows", "tiles", "binary64"])
def test_shared_equals_alone(search, gas, stencil):
    precision = 0 if search == "binary64" else 1
    kernel = {"rows": 3, "tiles": 2, "binary64": 0}[search]

    def make(n, flags):
        s, arrays = setup_of(n, gas)
        return kmc.Simulation(kmc.params_from_setup(s, precision=precision, stencil=stencil,
                                                    search_kernel=kernel, flags=flags), arrays)

    cases = [(n, f) for n in SIZES for f in (0, 1)]  # flags 1: no speed split
    alone = [make(*c) for c in cases]
    members = [make(*c) for c in cases] + [make(200003, 0)]
    group = kmc.Group(members)
    for m in members:
        group.budget(m, 3)
    for step in range(3):
        group.step(1)
        group.sync()
        for c, a, b in zip(cases, alone, members):
            a.step(1).sync()
            assert a.counts()[-1] == b.counts()[-1], (c, step)
            assert np.array_equal(a.partners(), b.partners()), (c, step)
    for c, a, b in zip(cases, alone, members):
        sa, la = a.state()
        sb, lb = b.state()
        assert all(np.array_equal(x.view(np.uint64), y.view(np.uint64)) for x, y in zip(sa, sb)), c
        assert np.array_equal(la, lb), c
    group.close()
    for sim in alone + members:
        sim.close()
