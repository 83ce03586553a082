"""The work this framework is used for, as cases that can be timed and compared.

Every case goes through the public Python interface (``Simulation``,
``Ensemble``, ``SparseLattice`` and the ``bl_*`` calls of the network).  Kinds:

* ``cells``  the coupled step of plasma and cells: walls of a shear cell or a
  duct, a tube given as a wall mask, or Lees-Edwards shear.  A pass is ``steps``
  time steps and a read-out of the fields (to the GPU) and the cells (to the
  host), as a run that samples every few steps does.
* ``drive``  a host program that sets the cells, takes one step and reads the
  cells back, every step.
* ``sweep``  an ensemble of independent shear cells stepped together.
* ``plasma`` the lattice without cells, ``vessel`` the indexed lattice of a
  vessel network: ``steps`` time steps and a read-out of the fields.
* ``train``  one epoch of the near-contact network: loss and gradient over the
  whole batch, one Adam step, and the weights.

The library reads out in FP64 what it computed in FP32 from populations stored
in ``store``; the outputs are kept in the type of the storage (the cells' state
and forces in FP32).

``exact`` is the method in plain FP64 torch: no code of this package but the
generators of the inputs.
"""
import functools
import math

import numpy as np
import torch

from paper_1005_2594_gb300 import bloodlb as bl
from paper_1005_2594_gb300 import rheology, workloads

STORE = {"f32": (bl.BL_STORE_F32, torch.float32, 4), "bf16": (bl.BL_STORE_BF16, torch.bfloat16, 2),
         "f16": (bl.BL_STORE_F16, torch.float16, 2)}
CELL = ("F", "T", "X", "q", "V", "L")


def _cells(name, geom, nx, ny, nz, hct, steps, R=7.0, store="f32", net=False):
    # R: the equatorial half-axis; the polar one is 3/7 of it, 1/3 in the tube and the sheared box
    return {"name": name, "kind": "cells", "geom": geom, "nx": nx, "ny": ny, "nz": nz, "hct": hct, "R": R,
            "steps": steps, "store": store, "net": net}


def listed():
    return [
        # the smallest suspension of the configurations: launches and latency
        _cells("cells_shear_32", "shear", 32, 32, 32, 0.047, 10, R=3.5),
        # a program that owns the cells' motion: state up, one step, forces down
        {"name": "drive_shear_128", "kind": "drive", "geom": "shear", "nx": 128, "ny": 128, "nz": 128, "hct": 0.30,
         "R": 7.0, "steps": 1, "store": "f32", "net": False},
        # the production shear cell (the benchmark's default workload)
        _cells("cells_shear_128", "shear", 128, 128, 128, 0.30, 10),
        # the precision workload's duct, plain storage and the 16-bit one
        _cells("cells_duct_256", "duct", 256, 256, 256, 0.31, 5),
        _cells("cells_duct_256_bf16", "duct", 256, 256, 256, 0.31, 5, store="bf16"),
        # the arteriole (odd cross-section, dense, soft wall) with the near-contact network on
        _cells("cells_tube_101_net", "tube", 64, 101, 101, 0.42, 20, R=5.5, net=True),
        # the rheology box: Lees-Edwards shear, dense suspension, small lattice
        _cells("cells_le_128x40", "le", 128, 40, 40, 0.44, 20, R=5.5),
        # a rheology sweep: uneven shear cells stepped as one ensemble
        {"name": "sweep_16", "kind": "sweep", "members": 16, "steps": 10, "store": "f32"},
        # plasma alone: a driven duct beyond the caches, and a ragged box at another tau, 16-bit storage
        {"name": "plasma_192", "kind": "plasma", "nx": 192, "ny": 192, "nz": 192, "tau": 1.0, "steps": 10,
         "store": "f32"},
        {"name": "plasma_150x77x63", "kind": "plasma", "nx": 150, "ny": 77, "nz": 63, "tau": 0.8, "steps": 20,
         "store": "f16"},
        # a vessel loop whose lumen fills 6 % of its box
        {"name": "vessel_1024x384x96", "kind": "vessel", "nx": 1024, "ny": 384, "nz": 96, "r0": 24.0, "tau": 1.0,
         "steps": 10, "store": "f32"},
        # one training epoch on the augmented approach samples
        {"name": "train_39400", "kind": "train", "batch": 39400},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("cells", "cells", "cells", "drive", "sweep", "plasma", "vessel", "train"))
    store = rng.choice(("f32", "f32", "bf16", "f16"))
    if kind in ("cells", "drive"):
        geom = rng.choice(("shear", "duct", "tube", "le"))
        small = rng.random() < 0.3
        R = rng.choice((3.5, 4.0)) if small else rng.choice((5.5, 7.0))
        lo, hi = (24, 64) if small else (44, 200)
        nx, ny, nz = (_log(rng, lo, hi) for _ in range(3))
        if geom == "tube":
            nz = ny
        c = _cells("", geom, nx, ny, nz, round(rng.uniform(0.05, 0.35), 3), rng.randint(3, 12), R=R, store=store,
                   net=geom == "tube" and rng.random() < 0.5)
        del c["name"]
        return dict(c, kind=kind, steps=1 if kind == "drive" else c["steps"])
    if kind == "sweep":
        return {"kind": kind, "members": rng.randint(2, 16), "steps": 2 * rng.randint(1, 5), "store": store}
    tau = rng.choice((1.0, 1.0, 0.8, 0.65))
    if kind == "plasma":
        return {"kind": kind, "nx": _log(rng, 20, 220), "ny": _log(rng, 12, 180), "nz": _log(rng, 12, 180), "tau": tau,
                "steps": rng.randint(2, 20), "store": store}
    if kind == "vessel":
        nz = _log(rng, 24, 96)
        return {"kind": kind, "nx": _log(rng, 96, 1024), "ny": 4 * nz + rng.randint(0, 7), "nz": nz, "r0": nz / 4.0,
                "tau": tau, "steps": rng.randint(2, 20), "store": store}
    return {"kind": kind, "batch": _log(rng, 500, 80000)}


# ---------------------------------------------------------------------------
# inputs


def _seed(case, seed):
    return (int(seed) * 1000003 + sum(ord(ch) for ch in repr(sorted((k, v) for k, v in case.items() if k != "name"))))


def _suspension(geom, nx, ny, nz, hct, R, seed, U=0.02):
    """params, wall mask or None, cell states X, q, V, L"""
    rng = np.random.default_rng(seed % (1 << 32))
    mask, inside = None, None
    if geom == "shear":
        p = workloads.base_params(nx, ny, nz, periodic=(1, 1, 0), R=(R, 3.0 / 7.0 * R), eps=1.0,
                                  wall_vel={4: (-U, 0.0, 0.0), 5: (U, 0.0, 0.0)})
    elif geom == "duct":
        p = workloads.base_params(nx, ny, nz, periodic=(1, 0, 0), R=(R, 3.0 / 7.0 * R), eps=1.0, g=(1e-6, 0.0, 0.0),
                                  body_force_on_cells=1)
    else:
        # cells of Sec. IV: the coupling half-axes are 11/12 of the potential's
        sig = (R * 12.0 / 11.0, R * 4.0 / 11.0)
        p = workloads.base_params(nx, ny, nz, periodic=(1, 1, 1), R=(R, R / 3.0), sigma=sig, eps=0.05,
                                  eps_w=0.005, g=(8e-6 if geom == "tube" else 0.0, 0.0, 0.0),
                                  body_force_on_cells=1 if geom == "tube" else 0)
    vol, lumen = workloads.cell_volume(p), float(nx * ny * nz)
    if geom == "tube":
        radius, c = ny / 2.0 - 4.0, (ny - 1) / 2.0
        mask, lumen = workloads.tube_mask(p, radius), math.pi * radius ** 2 * nx

        def inside(x):
            return np.hypot(x[:, 1] - c, x[:, 2] - c) + R + 1.0 < radius
    else:
        lo = np.array([0.0 if p["periodic"][k] else R + 2.5 for k in range(3)])
        hi = np.array([1e9 if p["periodic"][k] else (nx, ny, nz)[k] - 1.0 - R - 2.5 for k in range(3)])
        if geom == "le":
            lo[0], hi[0] = rheology.le_reflect_distance(p), nx - 1.0 - rheology.le_reflect_distance(p)

        def inside(x):
            return np.all((x >= lo) & (x <= hi), axis=1)

    n = max(1, int(round(hct * lumen / vol)))
    while True:
        try:
            # neighbours nearer than 1.6 polar diameters would start far inside
            # each other: fewer cells then (the same number for every seed)
            X, _ = workloads.fcc_cells(p, n, 0, inside)
            if n == 1 or _nearest(X, (nx, ny, nz), p["periodic"]) > 1.6 * 2.0 * p["R_par"]:
                X, q = workloads.fcc_cells(p, n, seed % (1 << 32), inside)
                break
        except ValueError:
            pass
        n = max(1, int(0.85 * n)) if n > 1 else 0
        if n == 0:
            X, q = np.array([[nx / 2.0, ny / 2.0, nz / 2.0]]), workloads.random_axes_and_quaternions(rng, 1)[1]
            n = 1
            break
    V = rng.uniform(-0.005, 0.005, (n, 3))
    L = rng.uniform(-0.001, 0.001, (n, 3)) * (p["rho_p"] * vol * R * R / 5.0)
    return p, mask, X, q, V, L


def _nearest(X, dims, per):
    best = 1e30
    for i0 in range(0, min(len(X), 1024), 512):  # (a lattice start: a part of it shows its spacing)
        d = X[i0:i0 + 512, None, :] - X[None, :, :]
        for k in range(3):
            if per[k]:
                d[..., k] -= dims[k] * np.round(d[..., k] / dims[k])
        r2 = (d * d).sum(axis=-1)
        r2[r2 == 0.0] = 1e30
        best = min(best, float(r2.min()))
    return math.sqrt(best)


LE_U = 0.0192
# the near-contact network is used inside these gaps and relative speeds
NET_RANGE = (0.3, 2.0, 0.0, 0.03)


def _network(seed):
    """weights and standardisation of a trained network's size and spread"""
    rng = np.random.default_rng((seed + 17) % (1 << 32))
    theta = []
    for rows, cols in ((64, 14), (64, 1), (64, 64), (64, 1), (6, 64), (6, 1)):
        lim = 1.0 / math.sqrt(cols) if cols > 1 else 0.02
        theta.append(rng.uniform(-lim, lim, rows * cols))
    norm = np.concatenate([np.zeros(14), [5.0] * 3 + [0.5] * 4 + [1.0] + [0.01] * 3 + [0.002] * 3, np.zeros(6),
                           [1e-3] * 3 + [3e-3] * 3])
    return np.concatenate(theta), norm


def _members(case, seed):
    rng = np.random.default_rng(seed % (1 << 32))
    out = []
    for k in range(case["members"]):
        n = (48, 64, 80, 96)[k % 4]
        out.append(_suspension("shear", n, n, n, (0.10, 0.30, 0.20)[(k // 4 + k) % 3], 7.0, seed + 101 * k,
                               U=float(rng.uniform(0.005, 0.05))))
    return out


def _plasma(case, seed):
    """params and the populations of a wavy flow between moving walls, driven by a body force"""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    rng = np.random.default_rng(seed % (1 << 32))
    p = workloads.base_params(nx, ny, nz, periodic=(1, 1, 0), g=(1e-5, 0.0, 0.0),
                              wall_vel={4: (-0.02, 0.0, 0.0), 5: (0.02, 0.01, 0.0)})
    p["tau"] = case["tau"]
    a, ph = rng.uniform(0.002, 0.02, 3), rng.uniform(0.0, 2.0 * math.pi, 3)
    ax = [torch.arange(m, dtype=torch.float64, device="cuda") * (2.0 * math.pi / m) for m in (nx, ny, nz)]
    u = [(a[k] * torch.sin(ax[(k + 1) % 3].view([-1 if d == 2 - (k + 1) % 3 else 1 for d in range(3)]) + ph[k]))
         .expand(nz, ny, nx) for k in range(3)]
    rho = 1.0 + 1e-3 * torch.cos(ax[0]).view(1, 1, -1).expand(nz, ny, nx)
    return p, rho, u


@functools.lru_cache(maxsize=2)
def _vessel_mask(nx, ny, nz, r0):
    return workloads.vessel_loop(nx, ny, nz, r0=r0, h=ny / 4.0)[0]


def _vessel(case, seed):
    rng = np.random.default_rng(seed % (1 << 32))
    # plasma at rest, set in motion by the body force and a part of the wall that slides
    p = workloads.base_params(case["nx"], case["ny"], case["nz"], g=(float(rng.uniform(0.5e-5, 2e-5)), 0.0, 0.0),
                              wall_vel={6: (float(rng.uniform(0.002, 0.01)), 0.0, 0.0)})
    p["tau"] = case["tau"]
    return p, _vessel_mask(case["nx"], case["ny"], case["nz"], case["r0"])


def _samples(case, seed):
    rng = np.random.default_rng(seed % (1 << 32))
    theta, norm = _network(seed)
    x = norm[14:28] * rng.normal(0.0, 1.0, (case["batch"], 14)) + norm[:14]
    y = norm[34:40] * np.tanh(x[:, :6] / norm[14:20]) * rng.uniform(0.5, 1.5, (case["batch"], 6))
    return theta, norm, x.astype(np.float32), y.astype(np.float32)


# ---------------------------------------------------------------------------
# state and pass


class _Out:
    """read-out buffers of one lattice, as a sampling program keeps them"""

    def __init__(self, N):
        self.rho = torch.zeros(N, dtype=torch.float64, device="cuda")
        self.u = torch.zeros((N, 3), dtype=torch.float64, device="cuda")
        self.owner = torch.zeros(N, dtype=torch.int32, device="cuda")


def _sim(case, p, mask, X, q, V, L):
    s = bl.Simulation(p, store_dtype=STORE[case["store"]][0], stream=torch.cuda.current_stream().cuda_stream,
                      wall_mask=mask)
    if case.get("geom") == "le":
        s.lees_edwards(LE_U)
    s.set_particles(X, q, V, L)
    return s


def prepare(case, seed):
    sd, st = _seed(case, seed), {"case": case}
    kind = case["kind"]
    if kind in ("cells", "drive"):
        p, mask, X, q, V, L = _suspension(case["geom"], case["nx"], case["ny"], case["nz"], case["hct"], case["R"], sd)
        st["sim"] = _sim(case, p, mask, X, q, V, L)
        st["state"] = {"X": X, "q": q, "V": V, "L": L}
        if case["net"]:
            theta, norm = _network(sd)
            st["net"] = bl.bl_mlp_create(torch.cuda.current_stream().cuda_stream)
            bl.bl_mlp_params_set(st["net"], theta, norm)
            bl.bl_mlp_attach_range(st["sim"].ctx, st["net"], *NET_RANGE)
        st["out"] = _Out(st["sim"].N)
    elif kind == "sweep":
        sims = [_sim(case, *m) for m in _members(case, sd)]
        st["ens"] = bl.Ensemble(sims, stream=torch.cuda.current_stream().cuda_stream)
        st["out"] = [_Out(s.N) for s in sims]
    elif kind == "plasma":
        p, rho, u = _plasma(case, sd)
        st["sim"] = bl.Simulation(p, store_dtype=STORE[case["store"]][0], stream=torch.cuda.current_stream().cuda_stream)
        pop = torch.empty((rho.numel(), 19), dtype=torch.float64, device="cuda")
        for r in range(19):
            pop[:, r] = _equilibrium(rho, u, r).reshape(-1)
        st["sim"].set_populations(pop.cpu().numpy())
        st["out"] = _Out(st["sim"].N)
    elif kind == "vessel":
        p, mask = _vessel(case, sd)
        st["sim"] = bl.SparseLattice(p, mask, store_dtype=STORE[case["store"]][0],
                                     stream=torch.cuda.current_stream().cuda_stream)
        st["out"] = _Out(st["sim"].N)
    else:
        theta, norm, x, y = _samples(case, sd)
        st["net"] = bl.bl_mlp_create(torch.cuda.current_stream().cuda_stream)
        bl.bl_mlp_params_set(st["net"], theta, norm)
        st["x"], st["y"] = torch.tensor(x, device="cuda"), torch.tensor(y, device="cuda")
    return st


def _fields(sim, o, dt):
    bl.bl_fields_get(sim.ctx, sim.N, o.rho, o.u, o.owner, on_device=True)
    return {"rho": o.rho.to(dt), "u": o.u.to(dt), "owner": o.owner}


def _state(a, dt):
    return {k: torch.from_numpy(a[k]).to(dt) for k in CELL}


def run(state):
    case = state["case"]
    kind, dt = case["kind"], STORE[case.get("store", "f32")][1]
    if kind == "cells":
        state["sim"].step(case["steps"])
        out = _fields(state["sim"], state["out"], dt)
        out.update(_state(state["sim"].particles(), dt))
        if case["geom"] == "le":
            out["P"] = torch.tensor(state["sim"].lees_edwards_momentum()[0], dtype=dt)
        return out
    if kind == "drive":
        s, c = state["sim"], state["state"]
        s.set_particles(c["X"], c["q"], c["V"], c["L"])
        s.step(1)
        state["state"] = s.particles()
        return _state(state["state"], dt)
    if kind == "sweep":
        e = state["ens"]
        e.step(case["steps"])
        f = [_fields(s, o, dt) for s, o in zip(e.sims, state["out"])]
        out = {k: torch.cat([x[k] for x in f]) for k in ("rho", "u", "owner")}
        c = [s.particles() for s in e.sims]
        out.update(_state({k: np.concatenate([x[k] for x in c]) for k in CELL}, dt))
        return out
    if kind == "plasma":
        state["sim"].step(case["steps"])
        out = _fields(state["sim"], state["out"], dt)
        return {"rho": out["rho"], "u": out["u"]}
    if kind == "vessel":
        o = state["out"]
        state["sim"].step(case["steps"])
        bl.bl_sparse_fields_get(state["sim"].h, state["sim"].N, o.rho, o.u, on_device=True)
        return {"rho": o.rho.to(dt), "u": o.u.to(dt)}
    loss, grad = bl.bl_mlp_grad(state["net"], state["x"], state["y"], want_grad=True)
    bl.bl_mlp_adam(state["net"], lr=1e-3)
    return {"loss": np.float32(loss), "grad": grad, "theta": bl.bl_mlp_params_get(state["net"])[0]}


def _pass_work(N, fluid, case, fields=True):
    # a step reads and writes each fluid node's 19 populations and reads a node
    # word; the read-out reads them once and writes rho, u and the owner
    s = STORE[case["store"]][2]
    read = N * (4.0 * s + 4.0) + 19.0 * s * fluid if fields else 0.0
    return {"bytes": case["steps"] * (38.0 * s * fluid + 4.0 * N) + read, "flops": case["steps"] * 250.0 * fluid}


def work(case):
    kind = case["kind"]
    if kind in ("cells", "drive"):
        N = float(case["nx"]) * case["ny"] * case["nz"]
        lumen = N * (math.pi * (0.5 - 4.0 / case["ny"]) ** 2 if case["geom"] == "tube" else 1.0)
        return _pass_work(N, (1.0 - case["hct"]) * lumen, case, fields=kind == "cells")
    if kind == "sweep":
        N = float(sum((48, 64, 80, 96)[k % 4] ** 3 for k in range(case["members"])))
        return _pass_work(N, 0.8 * N, case)
    if kind == "plasma":
        N = float(case["nx"]) * case["ny"] * case["nz"]
        return _pass_work(N, N, case)
    if kind == "vessel":
        N = float(case["nx"]) * case["ny"] * case["nz"]
        fluid = float((_vessel_mask(case["nx"], case["ny"], case["nz"], case["r0"]) == 0).sum())
        w = _pass_work(fluid, fluid, case)
        w["bytes"] += (N - fluid) * 4.0 * STORE[case["store"]][2]
        return w
    return {"bytes": case["batch"] * 80.0 + 5510 * 4.0 * 6, "flops": 6.0 * case["batch"] * 5376}


# ---------------------------------------------------------------------------
# the method in plain FP64

C = [(0, 0, 0)]
for _a in ((1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (1, -1, 0), (1, 0, 1), (1, 0, -1), (0, 1, 1), (0, 1, -1)):
    C += [_a, tuple(-v for v in _a)]
W = [1.0 / 3.0] + [1.0 / 18.0] * 6 + [1.0 / 36.0] * 12
OPP = [0] + [r + 1 if r % 2 else r - 1 for r in range(1, 19)]


def _dot(c, u):
    v = 0.0
    for k in range(3):
        if c[k]:
            v = v + c[k] * u[k]
    return v


def _equilibrium(rho, u, r):
    cu, uu = _dot(C[r], u), u[0] * u[0] + u[1] * u[1] + u[2] * u[2]
    return W[r] * rho * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * uu + cu * (4.5 * cu * cu - 4.5 * uu))


def _roll(a, c, sign=1):
    """a at x - sign c (periodic; walls close the other axes)"""
    return torch.roll(a, (sign * c[2], sign * c[1], sign * c[0]), dims=(0, 1, 2))


def _cross(a, b):
    return torch.stack([a[:, 1] * b[:, 2] - a[:, 2] * b[:, 1], a[:, 2] * b[:, 0] - a[:, 0] * b[:, 2],
                        a[:, 0] * b[:, 1] - a[:, 1] * b[:, 0]], dim=1)


def _rot(q):
    w, x, y, z = q.unbind(1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], dim=1).view(-1, 3, 3)


def _qmul(a, b):
    w, x, y, z = a.unbind(1)
    W_, X, Y, Z = b.unbind(1)
    return torch.stack([w * W_ - x * X - y * Y - z * Z, w * X + x * W_ + y * Z - z * Y,
                        w * Y - x * Z + y * W_ + z * X, w * Z + x * Y - y * X + z * W_], dim=1)


class _Exact:
    """Plasma and cells in FP64; owner: -1 fluid, -2 - w wall w, k cell k."""

    def __init__(self, p, mask=None, le=False, net=None):
        self.p, self.net, self.le, self.t = p, net, le, 0
        self.dims = (p["nx"], p["ny"], p["nz"])
        shape = self.dims[::-1]
        own = torch.full(shape, -1, dtype=torch.int32, device="cuda")
        for k in (2, 1, 0):  # an edge node takes the first walled axis
            if not p["periodic"][k]:
                own.select(2 - k, self.dims[k] - 1).fill_(-2 - (2 * k + 1))
                own.select(2 - k, 0).fill_(-2 - 2 * k)
        if mask is not None:
            m = torch.tensor(np.asarray(mask).reshape(shape), device="cuda").to(torch.int32)
            own = torch.where(m > 0, -1 - m, own)
        self.owner = own
        self.n = torch.zeros((19,) + shape, dtype=torch.float64, device="cuda")
        for r in range(19):
            self.n[r] = torch.where(own == -1, W[r] * p["rho0"], 0.0)
        self.P = 0.0
        self.np = 0

    def image(self, d):
        for k in range(3):
            if self.p["periodic"][k]:
                d[..., k] -= self.dims[k] * ((d[..., k] > 0.5 * self.dims[k]).double() -
                                             (d[..., k] < -0.5 * self.dims[k]).double())
        return d

    def xyz(self, node):
        nx, ny, _ = self.dims
        return torch.stack([node % nx, node // nx % ny, node // (nx * ny)], dim=1).double()

    def around(self, X, ext):
        """(cell, node) of every node within ext of the cell's nearest node, each once"""
        g = torch.arange(-ext, ext + 1, device="cuda")
        off = torch.stack(torch.meshgrid(g, g, g, indexing="ij"), dim=-1).view(-1, 3)
        for i0 in range(0, X.shape[0], 1024):
            xc = X[i0:i0 + 1024].round().long()[:, None, :] + off[None]
            ok = torch.ones(xc.shape[:2], dtype=torch.bool, device="cuda")
            for k in range(3):
                if self.p["periodic"][k]:
                    if 2 * ext + 1 > self.dims[k]:
                        ok &= (off[:, k] >= -(self.dims[k] // 2)) & (off[:, k] < self.dims[k] - self.dims[k] // 2)
                    xc[..., k] %= self.dims[k]
                else:
                    ok &= (xc[..., k] >= 0) & (xc[..., k] < self.dims[k])
            i, j = torch.nonzero(ok, as_tuple=True)
            xc = xc[i, j]
            yield i + i0, xc[:, 0] + self.dims[0] * (xc[:, 1] + self.dims[1] * xc[:, 2])

    def cells(self, X, q, V, L):
        t = lambda a: torch.tensor(np.asarray(a), dtype=torch.float64, device="cuda")
        first, self.np = self.np == 0, len(X)
        self.X, self.q, self.V, self.L = t(X), t(q), t(V), t(L)
        m, Rp, Ra = self.mass(), self.p["R_perp"], self.p["R_par"]
        self.I_body = torch.tensor([m * (Ra * Ra + Rp * Rp) / 5.0] * 2 + [2.0 * m * Rp * Rp / 5.0],
                                   dtype=torch.float64, device="cuda")
        self.Om = torch.linalg.solve(self.inertia(), self.L)
        self.PF, self.PT = torch.zeros_like(self.X), torch.zeros_like(self.X)
        self.place(first)

    def mass(self):
        return self.p["rho_p"] * 4.0 / 3.0 * math.pi * self.p["R_perp"] ** 2 * self.p["R_par"]

    def inertia(self):
        R = _rot(self.q)
        return R @ (self.I_body[:, None] * R.transpose(1, 2))

    def place(self, first):
        """single occupancy by first arrival; covered fluid is deleted, freed nodes are filled"""
        p, own = self.p, self.owner.view(-1)
        axis = _rot(self.q)[:, :, 2]
        low = torch.full_like(own, 2 ** 31 - 1)
        keep = torch.zeros_like(own, dtype=torch.bool)
        for cell, node in self.around(self.X, int(math.ceil(max(p["R_perp"], p["R_par"]))) + 1):
            d = self.image(self.xyz(node) - self.X[cell])
            par = (d * axis[cell]).sum(1)
            s = par * par / p["R_par"] ** 2 + ((d * d).sum(1) - par * par) / p["R_perp"] ** 2
            cell, node = cell[s <= 1.0].to(torch.int32), node[s <= 1.0]
            low.scatter_reduce_(0, node, cell, "amin")
            keep[node[own[node] == cell]] = not first
        new = torch.where((own <= -2) | keep, own, torch.where(low < 2 ** 31 - 1, low, -1))
        node = torch.nonzero(new != own).view(-1)
        old, now = own[node].long(), new[node].long()
        n = self.n.view(19, -1)
        c = torch.tensor(C, dtype=torch.float64, device="cuda")
        mom = torch.zeros((len(node), 3), dtype=torch.float64, device="cuda")  # given to the new owner
        fluid = old == -1
        mom[fluid] = n[:, node[fluid]].T @ c
        arm = self.image(self.xyz(node) - self.X[old.clamp(min=0)])
        u = self.V[old.clamp(min=0)] + _cross(self.Om[old.clamp(min=0)], arm)
        mom[~fluid] = p["rho0"] * u[~fluid]
        n[:, node[fluid]] = 0.0
        if not first:
            o = ~fluid
            self.PF.index_add_(0, old[o], -mom[o])
            self.PT.index_add_(0, old[o], -_cross(arm[o], mom[o]))
            g = now >= 0
            arm = self.image(self.xyz(node) - self.X[now.clamp(min=0)])
            self.PF.index_add_(0, now[g], mom[g])
            self.PT.index_add_(0, now[g], _cross(arm[g], mom[g]))
        free = now == -1
        for r in range(19):
            n[r, node[free]] = _equilibrium(p["rho0"], u[free].unbind(1), r)
        self.owner = new.view_as(self.owner)

    def potentials(self):
        p = self.p
        F, T = torch.zeros_like(self.X), torch.zeros_like(self.X)
        R = _rot(self.q)
        axis = R[:, :, 2]
        sp2, sq2, sw2 = p["sig_par"] ** 2, p["sig_perp"] ** 2, p["sig_w"] ** 2
        chi = (sp2 - sq2) / (sp2 + sq2)
        for i0 in range(0, self.np, 1024):
            D = self.image(self.X[None] - self.X[i0:i0 + 1024, None])
            i, j = torch.nonzero(((D * D).sum(-1) < p["r_cut"] ** 2) & ((D * D).sum(-1) > 0.0), as_tuple=True)
            d, i = D[i, j], i + i0
            ang = [axis[i].clone().requires_grad_(True), d.clone().requires_grad_(True)]
            r = ang[1].norm(dim=1)
            e = ang[1] / r[:, None]
            a, b, c = (e * ang[0]).sum(1), (e * axis[j]).sum(1), (ang[0] * axis[j]).sum(1)
            sig = 2.0 * p["sig_perp"] / torch.sqrt(
                1.0 - 0.5 * chi * ((a + b) ** 2 / (1.0 + chi * c) + (a - b) ** 2 / (1.0 - chi * c)))
            eps = p["eps"] * (1.0 - chi * chi * c * c) ** (-0.5 * p["nu"])
            phi = torch.where(r < sig, eps * (1.0 - r / sig) ** 2, 0.0).sum()
            do, dr = torch.autograd.grad(phi, ang)
            F.index_add_(0, i, dr)  # d = X_j - X_i: the force on i is + d phi / d d
            T.index_add_(0, i, -_cross(axis[i], do))
            if self.net is not None:
                self.correct(i, j, d, R, F, T)
        wall = self.owner <= -2
        near = torch.zeros_like(wall)
        for r in range(1, 19):
            near |= ~_roll(wall, C[r])
        surf = (wall & near).view(-1)
        if not bool(surf.any()):
            return F, T
        chi_w, reach = (sp2 - sq2) / (sp2 + sw2), math.sqrt(max(sp2, sq2) + sw2)
        for i, node in self.around(self.X, int(math.ceil(reach)) + 1):
            i, node = i[surf[node]], node[surf[node]]
            d = self.image(self.xyz(node) - self.X[i])
            ang = [axis[i].clone().requires_grad_(True), d.clone().requires_grad_(True)]
            r = ang[1].norm(dim=1)
            a = (ang[1] * ang[0]).sum(1) / r
            sig = math.sqrt(sq2 + sw2) / torch.sqrt(1.0 - chi_w * a * a)
            phi = torch.where(r < sig, p["eps_w"] * (1.0 - r / sig) ** 2, 0.0).sum()
            do, dr = torch.autograd.grad(phi, ang)
            F.index_add_(0, i, dr)
            T.index_add_(0, i, -_cross(axis[i], do))
        return F, T

    def correct(self, i, j, d, R, F, T):
        """the near-contact network on ordered pairs inside its range"""
        theta, norm = self.net
        p, axis = self.p, R[:, :, 2]
        Rp2, Rq2 = p["R_par"] ** 2, p["R_perp"] ** 2
        chi = (Rp2 - Rq2) / (Rp2 + Rq2)
        r = d.norm(dim=1)
        e = d / r[:, None]
        a, b, c = (e * axis[i]).sum(1), (e * axis[j]).sum(1), (axis[i] * axis[j]).sum(1)
        gap = r - 2.0 * p["R_perp"] / torch.sqrt(
            1.0 - 0.5 * chi * ((a + b) ** 2 / (1.0 + chi * c) + (a - b) ** 2 / (1.0 - chi * c)))
        body = lambda v: torch.einsum("nab,na->nb", R[i], v)
        dq = _qmul(self.q[i] * torch.tensor([1.0, -1.0, -1.0, -1.0], dtype=torch.float64, device="cuda"), self.q[j])
        dq = torch.where(dq[:, :1] < 0.0, -dq, dq)
        x = torch.cat([body(d), dq, gap[:, None], body(self.V[j] - self.V[i]), body(self.Om[j] - self.Om[i])], dim=1)
        sp = x[:, 8:11].norm(dim=1)
        lo, hi, slo, shi = NET_RANGE
        on = (gap >= lo) & (gap < hi) & (sp >= slo) & (sp <= shi)
        y = _net_forward(theta, (x - norm[:14]) / norm[14:28])[0] * norm[34:40] + norm[28:34]
        lab = lambda v: torch.einsum("nab,nb->na", R[i], v)
        F.index_add_(0, i[on], lab(y[:, :3])[on])
        T.index_add_(0, i[on], lab(y[:, 3:])[on])

    def step(self):
        p, own, n = self.p, self.owner, self.n
        fluid = own == -1
        rho = n.sum(0)
        rho1 = torch.where(fluid, rho, 1.0)
        g = [float(v) for v in p["g"]]
        u = []
        for k in range(3):
            j = sum(C[r][k] * n[r] for r in range(19) if C[r][k])
            u.append(torch.where(fluid, j / rho1 + 0.5 * g[k], 0.0))
        ug = u[0] * g[0] + u[1] * g[1] + u[2] * g[2]
        for r in range(19):
            cu, cg = _dot(C[r], u), _dot(C[r], g)
            src = W[r] * rho * (3.0 * (cg - ug) + 9.0 * cu * cg) if any(g) else 0.0
            n[r] = torch.where(fluid, n[r] - (n[r] - _equilibrium(rho, u, r)) / p["tau"] +
                               (1.0 - 0.5 / p["tau"]) * src, 0.0)
        if self.le:
            cross = self.shear(n, rho, u)
        flat = own.view(-1)
        if self.np:
            F, T = self.potentials()
            links, Fl, Tl = [], torch.zeros_like(self.X), torch.zeros_like(self.X)
            Z = torch.zeros((self.np, 6, 6), dtype=torch.float64, device="cuda")
            for r in range(1, 19):
                to = _roll(own, C[r], -1).reshape(-1)  # owner of x + c_r
                c = torch.tensor([C[r]], dtype=torch.float64, device="cuda")
                x = torch.nonzero((flat >= 0) & (to != -1) & (to != flat)).view(-1)  # contact links
                cell = flat[x].long()
                f = (-2.0 * W[r] * p["rho0"] * c).expand(len(x), 3)
                Fl.index_add_(0, cell, f)
                Tl.index_add_(0, cell, _cross(self.image(self.xyz(x) + 0.5 * c - self.X[cell]), f))
                x = torch.nonzero((flat == -1) & (to >= 0)).view(-1)  # bounce-back links
                cell = to[x].long()
                arm = self.image(self.xyz(x) + 0.5 * c - self.X[cell])
                f = 2.0 * n[r].reshape(-1)[x][:, None] * c
                b = torch.cat([c.expand(len(x), 3), _cross(arm, c.expand(len(x), 3))], dim=1)
                w = 6.0 * W[r] * rho.reshape(-1)[x]
                Fl.index_add_(0, cell, f)
                Tl.index_add_(0, cell, _cross(arm, f))
                Z.index_add_(0, cell, w[:, None, None] * b[:, :, None] * b[:, None, :])
                links.append((r, x, cell, b, w))
            m = self.mass()
            Fo = F + self.PF + (m * torch.tensor(g, dtype=torch.float64, device="cuda")
                                if p["body_force_on_cells"] else 0.0)
            To = T + self.PT
            I = self.inertia()
            A = Z.clone()
            A[:, :3, :3] += m * torch.eye(3, dtype=torch.float64, device="cuda")
            A[:, 3:, 3:] += I
            v = torch.linalg.solve(A, torch.cat([m * self.V + Fl + Fo, self.L + Tl + To], dim=1))
            drag = torch.einsum("nab,nb->na", Z, v)
            self.F, self.T = Fl - drag[:, :3] + Fo, Tl - drag[:, 3:] + To
            self.V, self.Om = v[:, :3].clone(), v[:, 3:].clone()
            self.L = torch.einsum("nab,nb->na", I, self.Om)
        new = torch.empty_like(n)
        new[0] = n[0]
        wv = torch.tensor(np.asarray(p["wall_vel"]), dtype=torch.float64, device="cuda")
        for r in range(1, 19):
            rb = OPP[r]
            src = _roll(own, C[r])  # owner of x - c_r
            vb = torch.zeros_like(rho)
            wall = src <= -2
            if bool(wall.any()):
                vb[wall] = (wv @ torch.tensor(C[r], dtype=torch.float64, device="cuda"))[(-2 - src[wall]).long()]
            new[r] = torch.where(src == -1, _roll(n[r], C[r]), n[rb] + 6.0 * W[r] * rho * vb)
        if self.np:
            for r, x, cell, b, w in links:  # C of the population returning along -c_r
                new[OPP[r]].view(-1)[x] -= w * (b * v[cell]).sum(1)
        if self.le:
            for x, r, val in cross:
                new[r, :, :, x] = val
        self.n = torch.where(fluid, new, 0.0)
        del new
        if self.np:
            if self.le:
                d = rheology.le_reflect_distance(p)
                lo, hi, vx = self.X[:, 0] + 0.5, self.dims[0] - 0.5 - self.X[:, 0], self.V[:, 0]
                self.V[:, 0] = torch.where(((lo < d) & (vx < 0)) | ((hi < d) & (vx > 0)), -vx, vx)
            self.X = self.X + self.V
            for k in range(3):
                if p["periodic"][k]:
                    self.X[:, k] %= self.dims[k]
            th = self.Om.norm(dim=1, keepdim=True)
            dq = torch.cat([torch.cos(0.5 * th), self.Om * torch.sin(0.5 * th) / th.clamp(min=1e-300)], dim=1)
            self.q = _qmul(dq, self.q)
            self.q = self.q / self.q.norm(dim=1, keepdim=True)
            self.PF, self.PT = torch.zeros_like(self.X), torch.zeros_like(self.X)
            self.place(False)
        self.t += 1

    def shear(self, n, rho, u):
        """Lees-Edwards: the populations that cross between x = nx - 1 and x = 0, and their momentum"""
        out, nz, D = [], self.dims[2], math.fmod(LE_U * self.t, self.dims[2])
        for r in range(1, 19):
            if not C[r][0]:
                continue
            up = C[r][0] == 1
            x, to, du, off = (-1, 0, -LE_U, D) if up else (0, -1, LE_U, -D)
            uu = [v[:, :, x] for v in u]
            moved = n[r, :, :, x] + _equilibrium(rho[:, :, x], uu[:2] + [uu[2] + du], r) - _equilibrium(rho[:, :, x], uu, r)
            self.P += float((0.5 if up else -0.5) * C[r][2] * (n[r, :, :, x] + moved).sum())
            k, w = math.floor(off), off - math.floor(off)
            s = torch.roll(moved, C[r][1], dims=1)
            at = lambda q: torch.roll(s, C[r][2] - q, dims=0)  # s at z - c_z + q
            out.append((to, r, (1.0 - w) * at(k) + w * at(k + 1)))
        return out

    def read(self):
        fluid = self.owner == -1
        rho = self.n.sum(0)
        rho1 = torch.where(fluid, rho, 1.0)
        u = torch.stack([torch.where(fluid, sum(C[r][k] * self.n[r] for r in range(19) if C[r][k]) / rho1 +
                                     0.5 * float(self.p["g"][k]), 0.0).view(-1) for k in range(3)], dim=1)
        return {"rho": rho.view(-1), "u": u}


def _net_forward(theta, x):
    k, w = 0, []
    for rows, cols in ((64, 14), (64, 1), (64, 64), (64, 1), (6, 64), (6, 1)):
        w.append(theta[k:k + rows * cols].view(rows, cols) if cols > 1 else theta[k:k + rows])
        k += rows * cols
    h1 = torch.tanh(x @ w[0].T + w[1])
    h2 = torch.tanh(h1 @ w[2].T + w[3])
    return h2 @ w[4].T + w[5], w


def _exact_cells(case, m, net=None):
    p, mask, X, q, V, L = m
    e = _Exact(p, mask, le=case.get("geom") == "le", net=net)
    e.cells(X, q, V, L)
    if case["kind"] == "drive":
        e.cells(X, q, V, L)
    for _ in range(case["steps"]):
        e.step()
    out = e.read() if case["kind"] != "drive" else {}
    out.update({k: getattr(e, k) for k in CELL})
    if case.get("geom") == "le":
        out["P"] = e.P
    return out


def exact(case, seed):
    sd, kind = _seed(case, seed), case["kind"]
    d64 = lambda a: torch.tensor(np.asarray(a, dtype=np.float32).astype(np.float64), device="cuda")
    if kind in ("cells", "drive"):
        m = _suspension(case["geom"], case["nx"], case["ny"], case["nz"], case["hct"], case["R"], sd)
        return _exact_cells(case, m, [d64(a) for a in _network(sd)] if case["net"] else None)
    if kind == "sweep":
        out = [_exact_cells(case, m) for m in _members(case, sd)]
        return {k: torch.cat([o[k] for o in out]) for k in ("rho", "u") + CELL}
    if kind in ("plasma", "vessel"):
        if kind == "plasma":
            p, rho, u = _plasma(case, sd)
            e = _Exact(p)
            for r in range(19):
                e.n[r] = torch.where(e.owner == -1, _equilibrium(rho, u, r), 0.0)
        else:
            p, mask = _vessel(case, sd)
            e = _Exact(p, mask)
        for _ in range(case["steps"]):
            e.step()
        return e.read()
    theta, norm, x, y = (d64(a) for a in _samples(case, sd))
    theta.requires_grad_(True)
    out = _net_forward(theta, (x - norm[:14]) / norm[14:28])[0]
    loss = (((out - (y - norm[28:34]) / norm[34:40]) ** 2).sum(1)).mean()
    g = torch.autograd.grad(loss, theta)[0]
    # Adam's first step: m / (1 - b1) = g, v / (1 - b2) = g^2
    return {"loss": loss.detach(), "grad": g, "theta": (theta - 1e-3 * g / (g.abs() + 1e-8)).detach()}
