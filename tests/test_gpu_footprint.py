"""Device memory of a lattice without cells: 19 populations and, per node, the
owner, the claim word, the neighbour word, the neighbour-cell word and the
pending velocity (4 + 4 + 4 + 4 + 16 bytes); what only cells need comes with
them and goes with them."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__

    __graft_entry__.build()
    import torch

    torch.cuda.init()
    yield


@pytest.mark.parametrize("store,size", [(0, 4), (1, 2)])
def test_bytes_per_node_without_cells(store, size):
    import numpy as np
    import torch

    from paper_1005_2594_gb300 import bloodlb as bl
    from paper_1005_2594_gb300 import workloads

    n = 192
    p = workloads.base_params(n, n, n)
    X, q = np.array([[12.0, 15.0, 20.0], [20.0, 30.0, 24.0]]), np.tile([1.0, 0.0, 0.0, 0.0], (2, 1))
    warm = bl.Simulation(workloads.base_params(40, 40, 40), store_dtype=store)
    warm.step(2)  # (what the first use of a kernel takes once)
    warm.set_particles(X, q)
    warm.step(3)
    warm.close()
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    sim = bl.Simulation(p, store_dtype=store)
    sim.step(2)
    sim.sync()
    used = free0 - torch.cuda.mem_get_info()[0]
    # allocations are rounded up to 2 MiB each: 64 MiB covers them and the graph
    limit = (19 * size + 32) * n ** 3 + (64 << 20)
    assert used <= limit, (used / n ** 3, limit / n ** 3)
    # cells come and go
    sim.set_particles(X, q)
    sim.step(3)
    sim.sync()
    sim.set_particles(np.zeros((0, 3)), np.zeros((0, 4)))
    sim.step(3)
    sim.sync()
    assert free0 - torch.cuda.mem_get_info()[0] <= limit
    sim.close()
