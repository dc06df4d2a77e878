"""The tiled search where a warp's 32 particles fall into several short runs: columns of a few
particles between reflecting walls, whose first tiles follow their rows through the same
shared-memory records.  Pair lists equal the thread-per-particle search's at every step, and
the oracle's at the first."""
import numpy as np
import pytest

import kmc_inputs as ki
import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1310_3437_gb300 as kmc  # noqa: E402


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n,width,steps", [(4096, 1.0, 12), (262139, 8.0, 4)])
def test_short_runs(n, width, steps, precision):
    walls = (ki.REFLECT,) * 3
    s = ki.equilibrium_setup(n=n, seed=n, d0=0.01, dt=0.003).with_(
        box=(0.12, width, width), bc=walls, piston_x0=0.12)
    rng = np.random.default_rng(n)
    arrays = [rng.random(n) * b for b in s.box] + [rng.standard_normal(n) for _ in range(3)]
    # flags 1: no speed split, every pair is a slow one
    sims = [kmc.Simulation(kmc.params_from_setup(s, precision=precision, search_kernel=kernel, flags=1),
                           arrays) for kernel in (2, 1)]
    pi, pj, _, _ = oracle.candidate_pairs(s, oracle.State(arrays))
    for step in range(steps):
        tiles, walk = ([sim.step(1).sync(), sim.edges()][1] for sim in sims)
        assert np.array_equal(tiles, walk), step
        if step == 0:
            assert len(tiles) > n // 50 and np.array_equal(tiles, np.stack([pi, pj], axis=1))
    for sim in sims:
        sim.close()
