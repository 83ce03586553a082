"""Separations near half a period, against the oracle: the periodic image is
the nearest one of the exact separation, not of the positions rounded to
nodes.  A period may be as short as 2 max(R) + 4, where cells in contact and
cells that hand a node over can be half a period apart.
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


# axis: the axis on which the cells lie just over half a period apart; period:
# even (the rounded separation can be half a period exactly) or odd
@pytest.mark.parametrize("period", [18, 19])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_pair_force_takes_the_nearest_image(axis, period):
    import oracle
    from paper_1005_2594_gb300 import bloodlb as bl
    from paper_1005_2594_gb300 import workloads

    shape = [20, 20, 20]
    shape[axis] = period
    p = workloads.base_params(*shape, R=(7.0, 3.0), eps=0.01)
    rng = np.random.default_rng(10 * axis + period)
    seen = 0
    while seen < 4:
        X = np.full((2, 3), 9.0) + rng.uniform(-0.4, 0.4, (2, 3))
        X[0, axis] = rng.integers(0, 4) + rng.uniform(0.5, 0.6)
        X[1, axis] = X[0, axis] + 0.5 * period + rng.uniform(0.05, 0.8 if period % 2 == 0 else 0.4)
        _, q = workloads.random_axes_and_quaternions(rng, 2)
        r = X[1] - X[0]
        r[axis] -= period
        if not np.abs(oracle.pair(p, r, oracle.axis(q[0]), oracle.axis(q[1]))[1]).max() > 1e-5:
            continue  # out of contact: another orientation
        seen += 1
        orc, sim = oracle.Oracle(p), bl.Simulation(p)
        orc.set_particles(X, q)
        sim.set_particles(X, q)
        orc.step(1)
        sim.step(1)
        fo, fg = orc.force_parts(), sim.force_parts()
        # the force of one pair in FP32 (the bar of the other parity tests)
        assert rel(fg["Fp"], fo["Fp"]) < 1e-5 and rel(fg["Tp"], fo["Tp"]) < 1e-5, (X, q)
        sim.close()


@pytest.mark.parametrize("axis", [1, 2])
@pytest.mark.parametrize("frac", [-0.3, 0.2])
def test_impulses_of_a_cell_set_half_a_period_away(axis, frac):
    """the nodes it leaves lie around half a period from its new centre: their
    lever arms are those of the nearest image of the exact position"""
    import oracle
    from paper_1005_2594_gb300 import bloodlb as bl
    from paper_1005_2594_gb300 import workloads

    p = workloads.base_params(20, 20, 20, R=(3.5, 1.5))
    rng = np.random.default_rng(axis)
    X = np.array([[6.2, 6.7, 7.1]])
    _, q = workloads.random_axes_and_quaternions(rng, 1)
    X2 = X.copy()
    X2[0, axis] = 16.0 + frac
    V = np.array([[0.013, -0.011, 0.017]])
    L = np.zeros((1, 3))
    orc, sim = oracle.Oracle(p), bl.Simulation(p)
    for s in (orc, sim):
        s.set_particles(X, q, V, L)
        s.set_particles(X2, q, V, L)
    PF, PT = orc.pending()
    got = sim.force_parts()
    assert rel(got["PF"], PF) < 1e-6 and rel(got["PT"], PT) < 1e-6  # (the bar of the other re-placements)
    sim.close()


@pytest.mark.parametrize("shape,periodic", [((20, 20, 20), (1, 1, 1)), ((21, 24, 20), (1, 1, 1)),
                                            ((44, 20, 22), (0, 1, 1)), ((40, 21, 24), (1, 0, 1))])
def test_cells_set_anywhere_leave_their_nodes(shape, periodic):
    """re-placements by any distance, owner maps exact and the impulses of the nodes left and entered"""
    import oracle
    from paper_1005_2594_gb300 import bloodlb as bl
    from paper_1005_2594_gb300 import workloads

    p = workloads.base_params(*shape, periodic=periodic, R=(3.5, 1.5))
    rng = np.random.default_rng(sum(shape))
    n = 3
    lo = np.array([0.0 if k else 6.0 for k in periodic])
    hi = np.array([s if k else s - 7.0 for s, k in zip(shape, periodic)])
    draw = lambda: (lo + rng.uniform(0.0, 1.0, (n, 3)) * (hi - lo), workloads.random_axes_and_quaternions(rng, n)[1])
    orc, sim = oracle.Oracle(p), bl.Simulation(p)
    X, q = draw()
    V, L = rng.uniform(-0.02, 0.02, (n, 3)), np.zeros((n, 3))
    for s in (orc, sim):
        s.set_particles(X, q, V, L)
    for _ in range(8):
        X, q = draw()
        for s in (orc, sim):
            s.set_particles(X, q, V, L)
        np.testing.assert_array_equal(sim.owner(), orc.owner())
        PF, PT = orc.pending()
        got = sim.force_parts()
        assert rel(got["PF"], PF) < 1e-6 and rel(got["PT"], PT) < 1e-6
    sim.close()


# spheres of radius 4 in a 12^3 box: cell 0 leaves a node that cell 1 covers
# through the boundary; on two axes they are just under half a period apart,
# and the positions rounded to nodes just over it
@pytest.mark.parametrize("X,v", [
    ([[1.3298, 8.7825, 0.3315], [8.4863, 0.7281, 7.4738]], [0.17137, -0.1396, 0.17188]),
    ([[3.3311, 1.3282, 2.8234], [10.4822, 8.4037, 6.6342]], [0.17203, 0.17472, -0.1352]),
    ([[3.3818, 3.3489, 10.8101], [10.4578, 10.4678, 2.5878]], [0.17462, 0.17309, -0.13397]),
])
def test_node_handed_over_through_the_boundary(X, v):
    import oracle
    from paper_1005_2594_gb300 import bloodlb as bl
    from paper_1005_2594_gb300 import workloads

    p = workloads.base_params(12, 12, 12, R=(4.0, 4.0), eps=0.0, r_cut=5.0)
    p["move_particles"] = 2
    X, V = np.array(X), np.array([v, [0.0, 0.0, 0.0]])
    q = np.tile([1.0, 0.0, 0.0, 0.0], (2, 1))
    orc, sim = oracle.Oracle(p), bl.Simulation(p)
    for s in (orc, sim):
        s.set_particles(X, q, V, np.zeros((2, 3)))
    before = orc.owner()
    orc.step(1)
    sim.step(1)
    after = orc.owner()
    assert ((before == 0) & (after == 1)).any()  # a direct change of owner
    np.testing.assert_array_equal(sim.owner(), after)
    sim.close()
