"""Branches of the cell kernels that ordinary suspensions seldom reach,
against the oracle: more than 64 cells near a node that changes hands (the
search through the cell list), a node between three cells and one between
cells and a wall (links given their term one by one), more than 512 nodes of
one cell that another cell's record covers first (the second pass over all
records), more than 4096 nodes in 128 rows of a cell (contact nodes found by
search).  Owner maps exact, forces and fields to the bar of the other parity
tests, 1e-5.
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


def rel(a, b):
    return np.abs(np.asarray(a) - np.asarray(b)).max() / np.abs(np.asarray(b)).max()


def crowd():
    """small overlapping spheroids of prescribed motion in a box with two walls: about 80 within reach of each, and
    fluid left between them"""
    from paper_1005_2594_gb300 import workloads

    p = workloads.base_params(20, 18, 22, periodic=(1, 1, 0), R=(2.0, 1.2), eps=0.0, r_cut=4.0,
                              wall_vel={4: (-0.01, 0.0, 0.0), 5: (0.0, 0.01, 0.0)})
    p["move_particles"] = 2
    rng = np.random.default_rng(3)
    n = 700
    # two thirds in a quarter of the box (many candidates there), the rest anywhere (fluid in between)
    X = rng.uniform(0.0, 1.0, (n, 3)) * np.array([20.0, 18.0, 17.0]) + np.array([0.0, 0.0, 2.0])
    X[: n * 2 // 3] = rng.uniform(0.0, 1.0, (n * 2 // 3, 3)) * np.array([8.0, 9.0, 9.0]) + np.array([3.0, 4.0, 2.0])
    _, q = workloads.random_axes_and_quaternions(rng, n)
    return p, X, q, rng.uniform(-0.04, 0.04, (n, 3)), np.zeros((n, 3))


def discs():
    """three large discs one above the other: one plane of fluid between the first two, the third in contact"""
    from paper_1005_2594_gb300 import workloads

    p = workloads.base_params(58, 58, 30, periodic=(1, 1, 0), R=(26.0, 3.0), eps=0.0, r_cut=27.0)
    X = np.array([[28.3, 29.1, 7.6], [28.9, 28.7, 14.4], [29.2, 29.4, 20.4]])
    q = np.tile([1.0, 0.0, 0.0, 0.0], (3, 1))
    V = np.array([[0.012, -0.004, 0.001], [-0.009, 0.006, -0.002], [0.003, 0.011, 0.002]])
    return p, X, q, V, np.array([[250.0, -180.0, 300.0], [-200.0, 150.0, 100.0], [120.0, 220.0, -260.0]])


def owners_beside_fluid(orc, N):
    """how many different cells each fluid node has links to, and whether it has one to a wall"""
    b = orc.boundary_links()
    node, own = b[:, 0], b[:, 2]
    pairs = np.unique(np.stack([node[own >= 0], own[own >= 0]], axis=1), axis=0)
    wall = np.zeros(N, bool)
    wall[node[own < -1]] = True
    return np.bincount(pairs[:, 0], minlength=N), wall


@pytest.mark.parametrize("tau", [1.0, 0.8])
def test_crowded_cells(tau):
    import oracle
    from paper_1005_2594_gb300 import bloodlb as bl

    p, X, q, V, L = crowd()
    p["tau"] = tau
    orc, sim = oracle.Oracle(p), bl.Simulation(p)
    for s in (orc, sim):
        s.set_particles(X, q, V, L)
    ncell, wall = owners_beside_fluid(orc, orc.N)
    assert (ncell >= 3).any() and ((ncell >= 2) & wall).any()
    reach = 2.0 * 2.0 + 2.0  # 2 max(R) + 2
    for _ in range(6):
        before, x = orc.owner(), orc.particles()["X"]
        orc.step(1)
        sim.step(1)
        after = orc.owner()
        left = (before >= 0) & (after != before)
        d = x[:, None, :] - x[np.unique(before[left])][None, :, :]
        d[..., 0] -= 20.0 * np.round(d[..., 0] / 20.0)
        d[..., 1] -= 18.0 * np.round(d[..., 1] / 18.0)
        assert ((d ** 2).sum(axis=-1) < (reach - 0.2) ** 2).sum(axis=0).max() > 64
        np.testing.assert_array_equal(sim.owner(), after)
        np.testing.assert_array_equal(sim.contact_links(), orc.contact_links())
    sim.sync()
    _compare(sim, orc)
    sim.close()


@pytest.mark.parametrize("tau", [1.0, 0.8])
def test_large_discs(tau):
    import oracle
    from paper_1005_2594_gb300 import bloodlb as bl

    p, X, q, V, L = discs()
    p["tau"] = tau
    orc, sim = oracle.Oracle(p), bl.Simulation(p)
    for s in (orc, sim):
        s.set_particles(X, q, V, L)
    ncell, _ = owners_beside_fluid(orc, orc.N)
    assert (ncell >= 2).sum() > 512
    z = np.arange(p["nz"])
    area = np.bincount(np.flatnonzero(orc.owner() == 0) // (58 * 58), minlength=z.size)
    assert 128 * np.sort(area)[-2:].sum() / 2 / 53 > 4096  # nodes in 128 rows near the middle plane
    assert len(orc.contact_links()) > 0
    for _ in range(4):
        orc.step(1)
        sim.step(1)
        np.testing.assert_array_equal(sim.owner(), orc.owner())
    sim.sync()
    _compare(sim, orc)
    sim.close()


def _compare(sim, orc):
    rho_o, u_o, own = orc.fields()
    rho_g, u_g, _ = sim.fields()
    fl = own == -1
    assert rel(u_g[fl], u_o[fl]) < 1e-5
    assert rel(rho_g[fl], rho_o[fl]) < 1e-5
    po, pg = orc.particles(), sim.particles()
    for k in ("F", "T", "X", "V"):
        assert rel(pg[k], po[k]) < 1e-5, k
