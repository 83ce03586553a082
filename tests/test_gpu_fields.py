"""The field read-out against sums in FP64 over the populations it reads.

k_fields sums in error-free FP32 parts (lb_moments.cuh).  Reference: numpy
FP64 sums over bl_populations_get minus its shift.  Bars, from the arithmetic:
the populations come back as fl64(f~ + alpha rho_bar), so a reference sum of 19
is off by at most 19 half-ulps of alpha rho_bar <= rho_bar / 3 plus the sum's
own roundings, below 40 2^-53 rho_bar together; the read-out's own error is a
few ulps of its values, the populations being below 0.1 rho_bar here: 1e-14
rho_bar for rho, 1e-14 for u = j / rho.
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


# rho0 1e-25 puts the populations below the range of the split sums (2^-60):
# the plain FP64 sums; 33 x 9 x 7 leaves a partial warp and a partial block
@pytest.mark.parametrize("rho0", [1.0, 1e-9, 1e-25])
@pytest.mark.parametrize("store", [0, 1])
@pytest.mark.parametrize("steps", [0, 1])  # both layouts of the stored populations
def test_fields_match_sums_of_the_populations(rho0, store, steps):
    from paper_1005_2594_gb300 import bloodlb as bl
    from paper_1005_2594_gb300 import workloads

    p = workloads.base_params(33, 9, 7, periodic=(1, 1, 0), g=(2e-5, 0.0, -1e-5))
    p["rho0"] = rho0
    N = 33 * 9 * 7
    rng = np.random.default_rng(4)
    pop = rho0 * W * (1.0 + rng.uniform(-0.1, 0.1, (N, 19)) * 10.0 ** rng.uniform(-6, 0, (N, 19)))
    pop[5] = rho0 * W  # a node at rest: exact zeros
    sim = bl.Simulation(p, store_dtype=store)
    sim.set_populations(pop)
    sim.step(steps)
    rho, u, own = sim.fields()
    f = sim.populations() - rho0 * W
    fl = own == -1
    m = f.sum(axis=1)[fl]
    ref = rho0 + m
    g = np.float32(p["g"]).astype(np.float64)
    assert np.abs(rho[fl] - ref).max() < 1e-14 * rho0
    assert np.abs(u[fl] - ((f @ C)[fl] / ref[:, None] + 0.5 * g)).max() < 1e-14
    assert not rho[~fl].any() and not u[~fl].any()
