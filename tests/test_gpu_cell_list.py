"""The cell list on both sides of the rule that chooses its build (one block
up to 4096 cells and 48 KB of bins and cells, else four kernels), against the
list formed on the host from the same positions: bins floor((X / N) nb), cells
in index order within a bin.  Exact.

58^3 nodes with bins of 2.5 nodes are 23^3 = 12167 bins; the block's shared
memory ends at 12256 bins and cells together (48 KB less the 128 bytes of its
scan), and all of 12257..12288 lie within 48 KB of bins and cells alone.
"""
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


def _host_list(X, dims, nb):
    b = np.clip(np.floor(X / np.array(dims, float) * nb).astype(int), 0, nb - 1)
    b = b[:, 0] + nb[0] * (b[:, 1] + nb[1] * b[:, 2])
    ids = np.argsort(b, kind="stable")
    return np.concatenate([[0], np.cumsum(np.bincount(b, minlength=int(np.prod(nb))))]), ids


@pytest.mark.parametrize("n,r_cut,bins", [
    (1, 2.5, 12167), (89, 2.5, 12167), (90, 2.5, 12167), (105, 2.5, 12167), (121, 2.5, 12167), (122, 2.5, 12167),
    (4095, 6.0, 729), (4096, 6.0, 729), (4097, 6.0, 729),
])
def test_list_matches_host(n, r_cut, bins):
    from paper_1005_2594_gb300 import bloodlb as bl
    from paper_1005_2594_gb300 import workloads

    shape = (58, 58, 58)
    p = workloads.base_params(*shape, R=(1.5, 1.2), eps=0.0, r_cut=r_cut)
    rng = np.random.default_rng(n)
    X = rng.uniform(0.0, 58.0, (n, 3))
    # a fifth of the coordinates on bin borders, one cell just below the period
    on = rng.random((n, 3)) < 0.2
    nb1 = int(58 // r_cut)
    X[on] = (rng.integers(0, nb1, on.sum()) * (58.0 / nb1)) % 58.0
    X[0] = np.nextafter(58.0, 0.0)
    _, q = workloads.random_axes_and_quaternions(rng, n)
    sim = bl.Simulation(p)
    sim.set_particles(X, q, rng.uniform(-0.01, 0.01, (n, 3)), np.zeros((n, 3)))
    for steps in (0, 1, 2):
        sim.step(steps)
        sim.sync()
        nb, start, ids = sim.cell_list()
        assert int(np.prod(nb)) == bins
        s_ref, ids_ref = _host_list(sim.particles()["X"], shape, nb)
        np.testing.assert_array_equal(start, s_ref)
        np.testing.assert_array_equal(ids, ids_ref)
    sim.close()
