"""The indexed lattice's rows (words, segments, table nodes) against the dense
lattice, bit for bit: the same FP32 arithmetic in the same order on the same
geometry, so every velocity and density agrees exactly.  The geometries are
the ones where the row index can go wrong: rows shorter than a warp, one node
wide, rows that end inside a warp, isolated nodes, several wall ids at one
node, fewer nodes than a warp, every axis periodic or walled.
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


@pytest.mark.parametrize("shape,periodic,fill,ids", [
    ((64, 10, 9), (1, 1, 1), 0.25, 1),   # runs cut by random walls
    ((37, 11, 6), (1, 1, 0), 0.10, 3),   # ragged rows, walls of three ids
    ((37, 8, 7), (0, 0, 0), 0.30, 2),    # walled on every axis
    ((1, 9, 8), (1, 1, 1), 0.2, 1),      # a row is one node: its own x neighbour
    ((2, 9, 8), (1, 1, 1), 0.2, 2),      # both x neighbours are one node
    ((5, 3, 2), (1, 1, 1), 0.3, 1),      # fewer nodes than a warp
    ((160, 6, 5), (1, 1, 1), 0.0, 1),    # no wall: long rows, only their ends wrap
    ((70, 6, 5), (1, 1, 1), 0.9, 2),     # isolated nodes
])
@pytest.mark.parametrize("store,tau", [(0, 1.0), (0, 0.8), (2, 1.0)])
def test_rows_match_dense_lattice(shape, periodic, fill, ids, store, tau):
    from paper_1005_2594_gb300 import bloodlb as bl
    from paper_1005_2594_gb300 import workloads

    rng = np.random.default_rng(sum(shape) + ids)
    p = workloads.base_params(*shape, periodic=periodic, g=(1e-5, -2e-5, 0.0),
                              wall_vel={w: tuple(rng.uniform(-0.01, 0.01, 3)) for w in range(8)})
    p["tau"] = tau
    N = int(np.prod(shape))
    mask = np.where(rng.random(N) < fill, rng.integers(6, 6 + ids, N), 0).astype(np.uint8)
    dense = bl.Simulation(p, store_dtype=store, wall_mask=mask)
    own = dense.owner()
    fl = own == -1
    w = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)
    pop = np.zeros((N, 19))
    pop[fl] = w * (1.0 + rng.uniform(-0.02, 0.02, (fl.sum(), 19)))
    sparse = bl.SparseLattice(p, mask, store_dtype=store)
    assert sparse.n_fluid == fl.sum()
    dense.set_populations(pop)
    sparse.set_populations(pop)
    for steps in (1, 2, 5):  # both parities, single steps and replayed pairs
        dense.step(steps)
        sparse.step(steps)
        rho_d, u_d, _ = dense.fields()
        rho_s, u_s = sparse.fields()
        np.testing.assert_array_equal(u_s[fl], u_d[fl])
        np.testing.assert_array_equal(rho_s[fl], rho_d[fl])
        np.testing.assert_array_equal(sparse.populations()[fl], dense.populations()[fl])
        wd, ws = dense.wall_momentum(), sparse.wall_momentum()
        # sums of at most 18 N FP32 terms below 0.4 in different orders
        assert np.abs(wd - ws).max() <= 18 * N * 0.4 * 2.0 ** -23
