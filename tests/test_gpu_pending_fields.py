"""The field read-out beside moving cells: between steps the moving-boundary
terms of the last bounces are pending, and the read-out adds them as it reads
the populations, in every storage type and both layouts of the populations.

Reference: numpy FP64 sums over bl_populations_get, which gives the pending
terms to the stored populations first.  The populations behind both are the
same numbers, so the bars are those of the sums alone (19 half-ulps of
alpha rho_bar <= 1/3 in the reference, a few ulps in the read-out: 1e-14), and
the read-out before and after the terms are stored is the same bit for bit.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

W = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)
C = np.array([(0, 0, 0)] + [s * np.array(a) for a in ((1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (1, -1, 0), (1, 0, 1),
                                                    (1, 0, -1), (0, 1, 1), (0, 1, -1)) for s in (1, -1)])


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__

    __graft_entry__.build()
    import torch

    torch.cuda.init()
    yield


@pytest.mark.parametrize("tau", [1.0, 0.8])
@pytest.mark.parametrize("store", [0, 1, 2])
@pytest.mark.parametrize("steps", [1, 2])  # both layouts of the stored populations
def test_fields_add_the_pending_terms(steps, store, tau):
    from paper_1005_2594_gb300 import bloodlb as bl
    from paper_1005_2594_gb300 import workloads

    p, X, q = workloads.small_shear(seed=1031, n_cells=20)
    p["tau"], p["g"] = tau, (2e-5, 0.0, -1e-5)
    rng = np.random.default_rng(7)
    V, L = rng.uniform(-0.02, 0.02, X.shape), rng.uniform(-1.0, 1.0, X.shape)
    sim = bl.Simulation(p, store_dtype=store)
    sim.set_particles(X, q, V, L)
    sim.step(steps)
    first = sim.fields()
    again = sim.fields()  # a read-out leaves the state as it is
    f = sim.populations() - W
    after = sim.fields()
    for a, b, c in zip(first, again, after):
        np.testing.assert_array_equal(a, b)
        np.testing.assert_array_equal(a, c)
    rho, u, own = first
    fl = own == -1
    ref = 1.0 + f.sum(axis=1)[fl]
    g = np.float32(p["g"]).astype(np.float64)
    assert np.abs(rho[fl] - ref).max() < 1e-14
    assert np.abs(u[fl] - ((f @ C)[fl] / ref[:, None] + 0.5 * g)).max() < 1e-14
    assert not rho[~fl].any() and not u[~fl].any()
    # the terms are there to be added: fluid beside a cell moves with it
    assert np.abs(u[fl]).max() > 1e-3
    sim.close()
