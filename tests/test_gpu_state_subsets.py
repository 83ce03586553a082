"""bl_forces_get with some of its arrays left out: what is asked for equals the
full read-out, whichever arrays lie between, and the rest is not written."""
import itertools

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__

    __graft_entry__.build()
    import torch

    torch.cuda.init()
    yield


def test_any_subset_of_the_state():
    from paper_1005_2594_gb300 import bloodlb as bl
    from paper_1005_2594_gb300 import workloads

    p, X, q = workloads.small_shear(n_cells=7)
    rng = np.random.default_rng(0)
    sim = bl.Simulation(p)
    sim.set_particles(X, q, rng.uniform(-0.01, 0.01, X.shape), rng.uniform(-1.0, 1.0, X.shape))
    sim.step(3)
    keys = ("F", "T", "X", "q", "V", "L")
    full = sim.particles()
    for ask in itertools.product((False, True), repeat=6):
        got = {k: np.full_like(full[k], np.nan) for k, a in zip(keys, ask) if a}
        bl._check(sim.ctx, bl.lib().bl_forces_get(sim.ctx, *(bl._dp(got[k]) if k in got else None for k in keys)))
        for k in got:
            np.testing.assert_array_equal(got[k], full[k])
    sim.close()
