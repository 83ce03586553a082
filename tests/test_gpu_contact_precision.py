"""Rounding of the contact forces: 1728 pairs of cells in contact, each pair by
itself, against the potentials evaluated in extended precision (Eqs. phi,
epsilon, sigma and sigmaw from the same FP64 positions and axes).

Bar, from the arithmetic alone: with the separation, the shape function, the
contact distance and the overlap formed in FP64 and rounded to FP32 once each,
and the strength, the derivatives and the force in FP32, the same formulas
evaluated in numpy (every operation rounded, nothing fused) are off by 8.6e-8
of the force, root mean square, for pairs of this shape (8.5e-8 to 9.8e-8 for
the shapes of the workloads), and the torque by 6.1e-8 of F R_perp; with the
overlap's quotient and the contact distance formed in FP32 by 1.00e-7 and
6.4e-8.  Bars: 9.3e-8 for F, between the two (the sampling error of 1728 forces
is 2 %), and 7e-8 for T.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

R = (1.5, 4.5 / 7.0)  # (R_perp, R_par) as 7 : 3


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__

    __graft_entry__.build()
    import torch

    torch.cuda.init()
    yield


def pair_force(r, oi, oj, sig_perp, sig_par):
    """F and T on i in long double (eps = nu = 1, mu = 0)"""
    D = np.longdouble
    r, oi, oj = r.astype(D), oi.astype(D), oj.astype(D)
    dot = lambda a, b: (a * b).sum(axis=-1)
    sp2, sq2 = D(sig_par) ** 2, D(sig_perp) ** 2
    chi = (sp2 - sq2) / (sp2 + sq2)
    rl = np.sqrt(dot(r, r))
    rh = r / rl[:, None]
    a, b, c = dot(rh, oi), dot(rh, oj), dot(oi, oj)
    ap, am, dp, dm, e1 = a + b, a - b, 1 + chi * c, 1 - chi * c, 1 - (chi * c) ** 2
    S = 1 - chi / 2 * (ap ** 2 / dp + am ** 2 / dm)
    sigma = 2 * D(sig_perp) / np.sqrt(S)
    h, eps = 1 - rl / sigma, 1 / np.sqrt(e1)
    k = eps * h * rl / (sigma * S)
    pa, pb = k * chi * (ap / dp + am / dm), k * chi * (ap / dp - am / dm)
    pc = h * h * eps * chi ** 2 * c / e1 - k * chi ** 2 / 2 * ((ap / dp) ** 2 - (am / dm) ** 2)
    F = (-2 * eps * h / sigma)[:, None] * rh + (pa[:, None] * (oi - a[:, None] * rh) +
                                                pb[:, None] * (oj - b[:, None] * rh)) / rl[:, None]
    return F, -np.cross(oi, pa[:, None] * rh + pc[:, None] * oj), h


def test_pair_force_rounding():
    import oracle
    from paper_1005_2594_gb300 import bloodlb as bl
    from paper_1005_2594_gb300 import workloads

    m, d = 12, 8
    p = workloads.base_params(m * d, m * d, m * d, R=R, eps=1.0, r_cut=3.2)
    p["move_particles"] = 0
    rng = np.random.default_rng(11)
    n = m ** 3
    site = np.stack(np.meshgrid(*[np.arange(m)] * 3, indexing="ij"), -1).reshape(n, 3) * d + d / 2.0
    _, q = workloads.random_axes_and_quaternions(rng, 2 * n)
    o = np.array([oracle.axis(x) for x in q])
    u, _ = workloads.random_axes_and_quaternions(rng, n)
    # the contact distance along u, then an overlap of 1e-4 to 0.1
    chi = (R[1] ** 2 - R[0] ** 2) / (R[1] ** 2 + R[0] ** 2)
    a, b, c = (u * o[:n]).sum(-1), (u * o[n:]).sum(-1), (o[:n] * o[n:]).sum(-1)
    sig = 2.0 * R[0] / np.sqrt(1.0 - chi / 2 * ((a + b) ** 2 / (1 + chi * c) + (a - b) ** 2 / (1 - chi * c)))
    r = u * (sig * (1.0 - 10.0 ** rng.uniform(-4.0, -1.0, n)))[:, None]
    off = rng.uniform(-0.5, 0.5, (n, 3))
    X = np.concatenate([site + off - 0.5 * r, site + off + 0.5 * r])
    sim = bl.Simulation(p)
    sim.set_particles(X, q)
    sim.step(1)
    sim.sync()
    got = sim.force_parts()
    for i, j in ((slice(0, n), slice(n, 2 * n)), (slice(n, 2 * n), slice(0, n))):
        F, T, h = pair_force(X[j] - X[i], o[i], o[j], R[0], R[1])
        assert (h > 5e-5).all()
        f = np.sqrt((F ** 2).sum(-1))
        eF = np.sqrt(((got["Fp"][i] - F) ** 2).sum(-1)) / f
        eT = np.sqrt(((got["Tp"][i] - T) ** 2).sum(-1)) / (f * R[0])
        print("F rms %.3e max %.2e, T rms %.3e max %.2e" % tuple(float(v) for v in (
            np.sqrt((eF ** 2).mean()), eF.max(), np.sqrt((eT ** 2).mean()), eT.max())))
        assert np.sqrt((eF ** 2).mean()) < 9.3e-8
        assert np.sqrt((eT ** 2).mean()) < 7e-8
    sim.close()
