"""What this framework is used for, as cases to be measured.

A case is a dict of plain values.  ``prepare`` makes what a program holds
before the call (a lattice with its geometry, voltages and multigrid
hierarchy, a batch, or the tensors of a gradient call), ``run`` is one pass
through the public entry points, ``work`` what a pass cannot do without, and
``exact`` the same results from a plain FP64 torch restatement of the method
that shares no code with the library.

Kinds of case:

* ``steps``     nsteps time steps of one lattice, the induced charge and the
                fields, continuing from the state of the previous pass (a
                long simulation that samples its state now and then; it
                begins with charged layers and a few steps of flow), or with
                ``restart`` from the uncharged capacitor every time (one
                point of a parameter study)
* ``drive``     a time-dependent electrode voltage: new potentials, one step
                and the charge, every step
* ``batch``     many capacitors of uneven sizes advanced together
* ``gradient``  d Q / d (voltage, Debye length, diffusivities, occupancy)
* ``fields``    every observable of a lattice's state

Geometries: ``plates``, ``coax``, ``eof`` (plates with a tangential field),
``porous`` (spheres on a plate, solvent at rest), ``blobs`` (random solid
clusters of three electrodes, three ionic species).

Outputs keep the type in which the library computes them: potentials,
concentrations, charges and the FP64 form's populations are float64; the FP32
form's velocities and its gradients carry 24 bits and are handed on as float32.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1907_04732_gb300 import adjoint, lbe, workloads

_L_B = 1.44          # Bjerrum length of the electro-osmosis, porous and batched workloads
_TOL = {"fp32": 1e-13, "fp64": 1e-14}  # of a Poisson solve (1e-13 is the binding's default)
_WARM = 20           # steps behind a state that a pass continues from


# ---------------------------------------------------------------------------
# the cases
def listed():
    return [
        # the smallest lattice in use: a plate column in the plain FP64 form,
        # its charging curve sampled every 50 steps (launch latency)
        _case("plates_fp64", "steps", "plates", 4, 4, 64, "fp64", 50),
        # the same form on a coaxial capacitor (reference curve of the FP32 form)
        _case("coax_fp64", "steps", "coax", 128, 128, 4, "fp64", 4),
        # the plain FP64 form at the benchmark's size
        _case("eof_fp64", "steps", "eof", 64, 64, 256, "fp64", 2),
        # the FP32 form on a lattice that fits L2, driven by an alternating
        # voltage: a host call and a charge read-back per step
        _case("coax_drive_fp32", "drive", "coax", 128, 128, 4, "fp32", 8),
        # the benchmark's electro-osmosis lattice, a long run
        _case("eof_fp32", "steps", "eof", 64, 64, 256, "fp32", 25),
        # ragged sizes, three species with unequal valencies and diffusivities
        _case("blobs_fp32", "steps", "blobs", 61, 47, 53, "fp32", 10),
        # the porous electrode (solvent at rest), the first steps of a
        # charging run from the uncharged state
        _case("porous_fp32", "steps", "porous", 256, 256, 128, "fp32", 5, restart=True),
        # a large flow lattice: far beyond the caches
        _case("eof_large_fp32", "steps", "eof", 256, 256, 256, "fp32", 6),
        # a sweep over sizes, Debye lengths and voltages
        {"name": "batch_fp32", "kind": "batch", "count": 64, "steps": 2},
        # gradients for a small electrode: a design loop's inner call
        {"name": "gradient_crop", "kind": "gradient", "nx": 32, "ny": 32, "nz": 16, "spheres": 2, "rmin": 3.0,
         "rmax": 5.0, "steps": 40, "every": 10, "slots": 0},
        # gradients for a larger one within a memory budget (binomial checkpoints)
        {"name": "gradient_porous", "kind": "gradient", "nx": 128, "ny": 128, "nz": 64, "spheres": 40, "rmin": 5.0,
         "rmax": 9.0, "steps": 20, "every": 0, "slots": 6},
        # the observables that an analysis reads from one state
        {"name": "fields_fp32", "kind": "fields", "geometry": "eof", "nx": 64, "ny": 64, "nz": 256,
         "precision": "fp32"},
    ]


def _case(name, kind, geometry, nx, ny, nz, precision, steps, restart=False):
    return {"name": name, "kind": kind, "geometry": geometry, "nx": nx, "ny": ny, "nz": nz, "precision": precision,
            "steps": steps, "restart": restart}


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["steps", "steps", "steps", "steps", "drive", "batch", "gradient", "fields"])
    if kind == "batch":
        return {"kind": "batch", "count": _log_int(rng, 6, 60), "steps": rng.randint(1, 2)}
    if kind == "gradient":
        nx, ny, nz = _log_int(rng, 24, 128), _log_int(rng, 24, 128), _log_int(rng, 16, 64)
        steps = rng.randint(10, 20) if nx * ny * nz > 100000 else rng.randint(20, 40)
        revolve = rng.random() < 0.5
        return {"kind": "gradient", "nx": nx, "ny": ny, "nz": nz, "spheres": max(1, nx * ny * nz // 26000),
                "rmin": nz / 8.0, "rmax": nz / 5.0, "steps": steps, "every": 0 if revolve else rng.randint(4, 12),
                "slots": rng.randint(4, 8) if revolve else 0}
    precision = "fp64" if kind == "steps" and rng.random() < 0.35 else "fp32"
    geometry = rng.choice(["plates", "coax", "eof", "blobs"] + (["porous"] if precision == "fp32" else []))
    if geometry == "coax":
        nx = ny = _log_int(rng, 24, 160)
        nz = rng.randint(1, 8)
    elif geometry == "blobs":
        nx, ny, nz = (_log_int(rng, 12, 64) for _ in range(3))
    elif geometry == "porous":
        nx, ny, nz = _log_int(rng, 32, 224), _log_int(rng, 32, 224), _log_int(rng, 24, 112)
    else:
        side = 64 if precision == "fp64" else 224
        nx, ny, nz = _log_int(rng, 1, side), _log_int(rng, 1, side), _log_int(rng, 24, 256)
    c = {"kind": kind, "geometry": geometry, "nx": nx, "ny": ny, "nz": nz, "precision": precision}
    if kind != "fields":
        nodes = nx * ny * nz
        most = {"fp32": 24 if nodes < 1 << 20 else 6, "fp64": 40 if nodes < 1 << 13 else 2}[precision]
        c["steps"] = rng.randint(max(1, most // 3), most)
        c["restart"] = kind == "steps" and geometry in ("porous", "blobs") and rng.random() < 0.5
    return c


# ---------------------------------------------------------------------------
# inputs
def _spheres(nx, ny, nz, n, rmin, rmax, rng):
    """Node ids of a porous electrode: spheres in the lower half (periodic
    along x and y) joined to a plate at z = 0 (electrode 1), a counter plate
    at z = nz - 1 (electrode 2) behind at least two fluid layers."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    ids = torch.zeros((nz, ny, nx), dtype=torch.uint8, device=dev)
    ax = [torch.arange(k, device=dev, dtype=torch.float64) for k in (nz, ny, nx)]
    for _ in range(n):
        c = rng.uniform([0, 0, 0], [nz / 2.0, ny, nx])
        r = rng.uniform(rmin, rmax)
        dz = (ax[0] - c[0]).abs()
        dy = (ax[1] - c[1]).abs()
        dx = (ax[2] - c[2]).abs()
        dy, dx = torch.minimum(dy, ny - dy), torch.minimum(dx, nx - dx)
        ids |= (dz.square()[:, None, None] + dy.square()[:, None] + dx.square() <= r * r).to(torch.uint8)
    ids[nz - 3:] = 0
    ids[0] = 1
    ids[nz - 1] = 2
    return ids


def _charged(w, c):
    """Solute amounts around charged electrodes: each ion's Boltzmann
    distribution in a potential that decays over the Debye length from every
    electrode (so that forces and flow are those of a running simulation)."""
    nz, ny, nx = w.ids.shape
    if c["geometry"] == "coax":
        y, x = np.mgrid[0:ny, 0:nx]
        r = np.hypot(x - (nx - 1) / 2.0, y - (ny - 1) / 2.0)
        d = [(r - w.extra["r1"])[None], (w.extra["r2"] - r)[None]]
    else:
        z = np.arange(nz)[:, None, None]
        d = [z - 0.5, nz - 1.5 - z]
    mid = 0.5 * (w.psi[0] + w.psi[1])
    phi = sum((p - mid) * np.exp(-np.maximum(k, 0.0) / w.debye) for p, k in zip(w.psi, d))
    n = np.stack([b * np.exp(-z * phi) for b, z in zip(_bulk(w), w.z)])
    return np.broadcast_to(n, (2, nz, ny, nx)) * (w.ids == 0)


def _workload(c, seed):
    """(Workload, initial solute amounts or None) of a lattice case."""
    w, n = _lattice_inputs(c, seed)
    if n is None and c["geometry"] != "porous" and not c.get("restart"):
        n = _charged(w, c)
    return w, n


def _lattice_inputs(c, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    geo, nx, ny, nz = c["geometry"], c["nx"], c["ny"], c["nz"]
    volt = float(rng.uniform(0.05, 0.3))
    D = tuple(float(d) for d in rng.uniform(0.03, 0.08, size=2))
    if geo == "plates":
        w = workloads.plate_capacitor(nx, ny, nz, debye=float(rng.uniform(4, 12)), psi=(0.1, 0.1 + volt), D=D)
        return w.with_(flow=c["precision"] == "fp64"), None  # with and without the solvent
    if geo == "coax":
        half = min(nx, ny) / 2.0
        w = workloads.coax_capacitor(nx, ny, nz, r1=float(rng.uniform(0.12, 0.2)) * half, r2=0.8 * half,
                                     debye=float(rng.uniform(3, 8)), psi=(0.0, volt), D=D)
        return w, None
    if geo == "eof":
        w = workloads.eof_plates(nx, ny, nz, debye=float(rng.uniform(8, 24)), voltage=volt,
                                 ex=float(rng.uniform(5e-4, 2e-3)), D=D)
        return w, None
    if geo == "porous":
        n = max(1, round(200 * nx * ny / 65536))
        s = nz / 128.0
        ids = _spheres(nx, ny, nz, n, max(1.5, 6 * s), max(2.5, 12 * s), rng).cpu().numpy()
        return workloads.Workload("porous", ids, 2, (1, 1, 0), (0.0, volt), _L_B, float(rng.uniform(5, 12)), D=D,
                                  flow=False), None
    if geo == "blobs":
        ids = workloads.random_blobs(nx, ny, nz, 3, 0.12, seed)
        w = workloads.Workload("blobs", ids, 3, (1, 1, 1), tuple(float(v) for v in rng.uniform(-0.2, 0.2, size=3)),
                               _L_B, float(rng.uniform(5, 12)), tau=0.9, D=(0.05, 0.03, 0.06), z=(1.0, 2.0, -1.0),
                               e_app=(1e-3, 0.0, -5e-4))
        rho = np.array(_bulk(w))
        n = rho[:, None, None, None] * (1.0 + 0.1 * rng.standard_normal((3, nz, ny, nx)))
        return w, n * (ids == 0)
    raise ValueError(geo)


def _bulk(w):
    """Bulk concentrations: a 1:1 salt, or +1, +2, -1 neutral in the bulk."""
    rs = workloads.bulk_density(w.debye, w.bjerrum)
    return (rs, rs) if len(w.z) == 2 else (0.5 * rs, 0.25 * rs, rs)


class _State:
    pass


def _lattice(w, precision):
    p = lbe.params_for(w, precision=lbe.LBE_FP32 if precision == "fp32" else lbe.LBE_FP64, tol=_TOL[precision])
    for k, v in enumerate(_bulk(w)):
        p.rho_bulk[k] = v
    lat = lbe.Lattice(p)
    lat.set_geometry(w.ids, w.n_elec)
    lat.set_voltage(w.psi)
    return lat


def _drive(w, steps, seed):
    """Potentials of a driven capacitor: a sine around the workload's."""
    phase = 0.1 * (seed % 63)
    return [tuple(p * (1.0 + 0.2 * math.sin(0.3 * (t + 1) + phase)) for p in w.psi) for t in range(steps)]


def _gradient_inputs(c, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    ids = _spheres(c["nx"], c["ny"], c["nz"], c["spheres"], c["rmin"], c["rmax"], rng).cpu().numpy()
    psi = np.float32([0.0, rng.uniform(0.05, 0.2)])
    debye = np.float32(rng.uniform(5, 10))
    D = np.float32(rng.uniform(0.03, 0.08, size=2))
    return ids, psi, debye, D


def _batch_inputs(c, seed):
    """The sweep's sizes, with other voltages, Debye lengths and diffusivities."""
    rng = np.random.Generator(np.random.PCG64(seed))
    return [w.with_(debye=float(math.exp(rng.uniform(math.log(2.0), math.log(32.0)))),
                    psi=(0.0, float(rng.uniform(-0.5, 0.5))),
                    D=tuple(float(d) for d in rng.uniform(0.03, 0.08, size=2)))
            for w in workloads.batch_instances(c["count"])]


def prepare(case, seed):
    s = _State()
    s.case = case
    kind = case["kind"]
    if kind == "batch":
        s.w = _batch_inputs(case, seed)
        s.batch = lbe.Batch(s.w)
        s.batch.init()
        return s
    if kind == "gradient":
        ids, psi, debye, D = _gradient_inputs(case, seed)
        w = workloads.Workload("porous", ids, 2, (1, 1, 0), tuple(float(v) for v in psi), _L_B, float(debye),
                               D=tuple(float(v) for v in D), flow=False, steps=case["steps"])
        if case["slots"]:
            s.lat = _lattice(w, "fp32")
            s.budget = case["slots"] * 48 * w.nodes
            s.rho_to_debye = -2.0 * _bulk(w)[0] / w.debye
            s.dchi = torch.empty(w.nodes, dtype=torch.float64, device="cuda")
        else:
            s.spec = adjoint.ChargeSpec.from_workload(w, every=case["every"], tol=_TOL["fp32"])
            leaf = lambda a: torch.tensor(a, dtype=torch.float32, requires_grad=True)
            s.theta = leaf(np.concatenate([psi, [debye], D]))  # the optimiser's parameters
            s.chi = leaf((ids == 1) | (ids == 2))
        return s
    w, n = _workload(case, seed)
    s.lat = _lattice(w, case["precision"])
    s.lat.init()
    if n is not None and not case.get("restart"):
        s.lat.set_state(n=n)
    if not case.get("restart"):
        s.lat.step(_WARM)
    if kind == "drive":
        s.psi = _drive(w, case["steps"], seed)
    if kind == "fields":
        s.w = w
        s.ids = torch.as_tensor(w.ids, device="cuda")
    s.n0 = n
    return s


# ---------------------------------------------------------------------------
# one pass
def _fields(lat, flow=True):
    out = {"phi": lat.field(lbe.FIELD_PHI, device=True), "n": lat.field(lbe.FIELD_N, device=True)}
    if flow and lat.p.precision == lbe.LBE_FP32:
        out["u"] = lat.field(lbe.FIELD_U, device=True).float()
    elif flow:
        out["f"] = lat.field(lbe.FIELD_F, device=True)
    return out


def run(s):
    c = s.case
    kind = c["kind"]
    if kind == "steps":
        if c["restart"]:
            s.lat.init()
            if s.n0 is not None:  # concentrations that are not uniform
                s.lat.set_state(n=s.n0)
        s.lat.step(c["steps"])
        return {"charge": s.lat.charge(), **_fields(s.lat, s.lat.p.flow)}
    if kind == "drive":
        q = []
        for psi in s.psi:
            s.lat.set_voltage(psi)
            s.lat.step(1)
            q.append(s.lat.charge())
        return {"charge": np.array(q), **_fields(s.lat, s.lat.p.flow)}
    if kind == "batch":
        b = s.batch
        b.step(c["steps"])
        sizes = [w.nodes for w in s.w]
        phi = torch.empty(sum(sizes), dtype=torch.float64, device="cuda")
        n = torch.empty(2 * sum(sizes), dtype=torch.float64, device="cuda")
        at = 0
        for i, k in enumerate(sizes):
            lbe.lbe_batch_fields(b.b, i, lbe.FIELD_PHI, phi.data_ptr() + 8 * at, True)
            lbe.lbe_batch_fields(b.b, i, lbe.FIELD_N, n.data_ptr() + 16 * at, True)
            at += k
        return {"charge": b.charge(), "phi": phi, "n": n}
    if kind == "gradient":
        if c["slots"]:
            q = s.lat.adjoint_forward_budget(c["steps"], s.budget)
            g, dchi = s.lat.adjoint_backward([1.0, 0.0], 1, s.dchi)
            theta = [*g.dpsi[:2], g.drho_bulk * s.rho_to_debye, *g.dD[:2]]
            return {"charge": q, "theta": np.float32(theta), "chi": dchi.float()}
        q = adjoint.induced_charge(s.theta[:2], s.theta[2], s.theta[3:], s.chi, s.spec)
        theta, chi = torch.autograd.grad(q[0], (s.theta, s.chi))
        return {"charge": q.detach(), "theta": theta, "chi": chi}
    if kind == "fields":
        lat, w = s.lat, s.w
        out = _fields(lat)
        out["rho"] = lat.field(lbe.FIELD_RHO, device=True).float()
        out["f"] = lat.field(lbe.FIELD_F, device=True).float()
        out["qnode"] = lat.field(lbe.FIELD_QNODE, device=True)
        out["charge"] = lat.charge_device(torch.empty(w.n_elec, dtype=torch.float64, device="cuda"))
        static = torch.empty(w.n_elec, dtype=torch.float64, device="cuda")
        lbe.lbe_induced_charge_static(out["phi"].data_ptr(), s.ids.data_ptr(), w.shape, w.periodic, w.bjerrum,
                                      w.n_elec, static.data_ptr(), lat.stream)
        out["charge_static"] = static
        return out
    raise ValueError(kind)


# ---------------------------------------------------------------------------
# what a pass cannot do without: the state read and written once per step
# (populations, solute, potential, one geometry word) and the results written
# once; arithmetic of the link fluxes (18 links), the collision and one
# stencil of the potential per step
def _step_work(nodes, species, precision, flow):
    b = 8 if precision == "fp64" else 4
    byt = 2 * 19 * b * bool(flow) + 2 * 8 * species + 2 * 8 + 4
    return nodes * byt, nodes * (18 * 20 * species + 300 * bool(flow) + 40)


def work(case):
    c = case
    kind = c["kind"]
    if kind == "batch":
        nodes = sum(w.nodes for w in _batch_inputs(c, 0))
        byt, ops = _step_work(nodes, 2, "fp32", True)
        return {"bytes": c["steps"] * byt + 24 * nodes, "flops": c["steps"] * ops}
    nodes = c["nx"] * c["ny"] * c["nz"]
    if kind == "gradient":
        byt, ops = _step_work(nodes, 2, "fp32", False)
        return {"bytes": 2 * c["steps"] * byt + 4 * nodes, "flops": 3 * c["steps"] * ops}
    species = 3 if c["geometry"] == "blobs" else 2
    flow = c["geometry"] != "porous" and (c["geometry"] != "plates" or c["precision"] == "fp64")
    b = 8 if c["precision"] == "fp64" else 4
    if kind == "fields":  # the state read once; phi, n, qnode and u, rho, f written
        return {"bytes": nodes * (19 * b + 8 * species + 8 + 4 + 8 * (2 + species) + 23 * b),
                "flops": nodes * (18 * 20 * species + 60)}
    byt, ops = _step_work(nodes, species, c["precision"], flow)
    out = 8 + 8 * species + (19 * 8 if b == 8 else 3 * 4) * flow
    return {"bytes": c["steps"] * byt + out * nodes, "flops": c["steps"] * ops}


# ---------------------------------------------------------------------------
# the method in plain FP64 torch
_HALF = [(1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (1, -1, 0), (1, 0, 1), (1, 0, -1), (0, 1, 1), (0, 1, -1)]
_C = [(0, 0, 0)] + _HALF + [tuple(-a for a in c) for c in _HALF]
_W = [1 / 3] + [1 / 18 if sum(map(abs, c)) == 1 else 1 / 36 for c in _C[1:]]
_A0 = 1.0 + 2.0 * math.sqrt(2.0)


def _opp(i):
    return 0 if i == 0 else (i + 9 if i <= 9 else i - 9)


def _at(a, c):
    """a at r + c for every node r (the last three axes are z, y, x)."""
    move = [(-c[k], d) for k, d in ((0, -1), (1, -2), (2, -3)) if c[k]]
    return torch.roll(a, [m for m, _ in move], [d for _, d in move]) if move else a


class _Reference:
    """One lattice in FP64: link fluxes, BGK collision, cell-overlap
    advection, the potential of the modified Laplacian."""

    def __init__(self, w, ids, bulk):
        self.w = w
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.ids = torch.as_tensor(ids, device=dev).long()
        self.fluid = self.ids == 0
        self.bulk = bulk
        self.open = [None] + [self.fluid & _at(self.fluid, c) for c in _C[1:]]
        # link weights of the modified Laplacian: 1/3 and 1/6, doubled
        # between fluid and solid; links of a node to itself drop out
        self.lap_w = [None]
        nz, ny, nx = self.ids.shape
        diag = torch.zeros(self.ids.shape, dtype=torch.float64, device=dev)
        self.full_diag = torch.zeros_like(diag)  # self links included
        for c in _C[1:]:
            own = all(d == 0 or n == 1 for d, n in zip(c, (nx, ny, nz)))
            base = 1 / 3 if sum(map(abs, c)) == 1 else 1 / 6
            wt = base * torch.where(self.fluid != _at(self.fluid, c), 2.0, 1.0).double()
            self.full_diag += wt
            if own:
                wt = torch.zeros_like(wt)
            self.lap_w.append(wt)
            diag += wt
        self.diag = torch.where(self.fluid, diag, 1.0)
        # links that do not leave a non-periodic face
        self.inside = [None]
        for c in _C[1:]:
            ok = torch.ones(self.ids.shape, dtype=torch.bool, device=dev)
            for axis, (d, per) in enumerate(zip(c, w.periodic)):
                if d and not per:
                    ok.select(2 - axis, -1 if d > 0 else 0).fill_(False)
            self.inside.append(ok)
        self.n = torch.stack([b * self.fluid.double() for b in bulk])
        self.f = torch.stack([wi * self.fluid.double() for wi in _W])
        self.dense = None
        self.set_voltage(w.psi)

    # -- potential
    def set_voltage(self, psi):
        table = torch.tensor([0.0] + list(psi), dtype=torch.float64, device=self.ids.device)
        old = getattr(self, "phi", torch.zeros_like(self.diag))
        self.phi = torch.where(self.fluid, old, table[self.ids])
        self.solve()

    def lap(self, phi):
        out = torch.zeros_like(phi)
        for i, c in enumerate(_C[1:], 1):
            out += self.lap_w[i] * (_at(phi, c) - phi)
        return out

    def residual(self, phi, n):
        z = torch.tensor(self.w.z, dtype=torch.float64, device=n.device)
        rho = torch.einsum("k,kzyx->zyx", z, n)
        return torch.where(self.fluid, self.lap(phi) + 4.0 * math.pi * self.w.bjerrum * rho, 0.0)

    def minus_lap(self, x):
        """-lap x on fluid nodes for an x that vanishes on solid ones."""
        def pair(a, d):
            return torch.roll(a, 1, d) + torch.roll(a, -1, d)
        px, py, pz = pair(x, -1), pair(x, -2), pair(x, -3)
        near = (px + py + pz) / 3 + (pair(px, -2) + pair(px, -3) + pair(py, -3)) / 6
        return torch.where(self.fluid, self.full_diag * x - near, 0.0)

    def inverse(self, b):
        """x with -lap x = b on fluid nodes, 0 on solid ones."""
        if self.fluid.numel() <= 4096:
            if self.dense is None:
                at = self.fluid.reshape(-1).nonzero()[:, 0]
                e = torch.zeros((len(at), self.fluid.numel()), dtype=torch.float64, device=b.device)
                e[torch.arange(len(at), device=b.device), at] = 1.0
                rows = self.minus_lap(e.reshape((-1,) + self.fluid.shape)).reshape(len(at), -1)
                self.dense = at, torch.linalg.inv(rows[:, at])
            at, inv = self.dense
            x = torch.zeros(self.fluid.numel(), dtype=torch.float64, device=b.device)
            x[at] = inv @ b.reshape(-1)[at]
            return x.reshape(self.fluid.shape)
        x = torch.zeros_like(b)
        r = b.clone()
        stop = 1e-7 * (r / self.diag).abs().max()
        u = r / self.diag
        p = u.clone()
        gam = (r * u).sum()
        for k in range(5000):
            a = self.minus_lap(p)
            alpha = gam / (p * a).sum()
            x += alpha * p
            r -= alpha * a
            u = r / self.diag
            if k % 8 == 0 and not u.abs().max() > stop:
                break
            new = (r * u).sum()
            p = u + (new / gam) * p
            gam = new
        return x

    def solve(self):
        last = math.inf
        for _ in range(6):
            r = self.residual(self.phi, self.n)
            size = float((r / self.diag).abs().max())
            if size < 1e-16 or size > 0.1 * last:
                break
            last = size
            self.phi = self.phi + self.inverse(r)

    # -- one step
    def fluxes(self):
        w = self.w
        out = self.n.clone()
        F = torch.zeros((3,) + self.phi.shape, dtype=torch.float64, device=self.phi.device)
        for i, c in enumerate(_C[1:], 1):
            length = math.sqrt(sum(map(abs, c)))
            d = _at(self.phi, c) - self.phi - sum(e * k for e, k in zip(w.e_app, c))
            g = torch.zeros_like(self.phi)
            for k, z in enumerate(w.z):
                n0, n1 = self.n[k], _at(self.n[k], c)
                em = torch.exp(-z * d)
                # n1 e^{dmu} - n0 in the form that does not lose the difference
                diff = (n1 - n0) + n1 * torch.expm1(z * d)
                j = torch.where(self.open[i], -(w.D[k] / _A0) / length * 0.5 * (1.0 + em) * diff, 0.0)
                out[k] -= j
                g += torch.where(self.open[i], j * (_A0 / w.D[k]) + (n1 - n0) / length, 0.0)
            for a in range(3):
                if c[a]:
                    F[a] += c[a] * g
        return out, F / (2.0 * _A0)

    def gathered(self):
        f = [self.f[0]]
        for i, c in enumerate(_C[1:], 1):
            back = tuple(-a for a in c)
            f.append(torch.where(self.open[_opp(i)], _at(self.f[i], back), self.f[_opp(i)]))
        return torch.stack(f)

    def moments(self, F):
        f = self.gathered()
        rho = f.sum(0)
        m = torch.stack([sum(c[a] * f[i] for i, c in enumerate(_C) if c[a]) for a in range(3)])
        safe = torch.where(self.fluid, rho, 1.0)
        return f, rho, torch.where(self.fluid, (m + 0.5 * F) / safe, 0.0)

    def step(self):
        n, F = self.fluxes()
        if self.w.flow:
            f, rho, u = self.moments(F)
            om, guo = 1.0 / self.w.tau, 1.0 - 0.5 / self.w.tau
            uu, uF = (u * u).sum(0), (u * F).sum(0)
            new = torch.empty_like(f)
            for i, c in enumerate(_C):
                cu = c[0] * u[0] + c[1] * u[1] + c[2] * u[2]
                cF = c[0] * F[0] + c[1] * F[1] + c[2] * F[2]
                feq = _W[i] * rho * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * uu)
                new[i] = torch.where(self.fluid, f[i] - om * (f[i] - feq)
                                     + guo * _W[i] * (3.0 * (cF - uF) + 9.0 * cu * cF), 0.0)
            self.f = new
            n = self.advect(n, u)
        self.n = n
        self.solve()

    def advect(self, n, u):
        over = lambda s, v: 1.0 - v.abs() if s == 0 else (s * v).clamp(min=0.0)
        out = torch.zeros_like(n)
        for d in range(27):
            s = (d % 3 - 1, d // 3 % 3 - 1, d // 9 - 1)
            wt = over(s[0], u[0]) * over(s[1], u[1]) * over(s[2], u[2])
            if d == 13:
                out += wt * n
                continue
            goes = self.fluid & _at(self.fluid, s)
            share = torch.where(goes, wt, 0.0) * n
            out += _at(share, tuple(-a for a in s))
            out += torch.where(self.fluid & ~goes, wt, 0.0) * n
        return out

    # -- observables
    def charge_map(self):
        s = torch.zeros_like(self.phi)
        for i, c in enumerate(_C[1:], 1):
            s += torch.where(_at(self.fluid, c), self.lap_w[i] * (_at(self.phi, c) - self.phi), 0.0)
        return torch.where(self.fluid, 0.0, -s / (4.0 * math.pi * self.w.bjerrum))

    def charge(self):
        q = self.charge_map()
        return torch.stack([q[self.ids == e].sum() for e in range(1, self.w.n_elec + 1)])


def _reduced(w, geometry):
    """The part of a lattice that repeats: a column between plates, a slice
    of a coaxial capacitor; and how often it does."""
    nx, ny, nz = w.shape
    if geometry in ("plates", "eof"):
        return np.s_[:, :1, :1], nx * ny
    if geometry == "coax":
        return np.s_[:1], nz
    return np.s_[:], 1


class _Repeated:
    """The reference on the repeating part, its results spread over the lattice."""

    def __init__(self, w, geometry, n=None):
        part, self.times = _reduced(w, geometry)
        self.shape = w.ids.shape
        self.ref = _Reference(w, w.ids[part], _bulk(w))
        if n is not None:
            n = np.ascontiguousarray(n[(slice(None),) + (part if isinstance(part, tuple) else (part,))])
            self.ref.n = torch.as_tensor(n, device=self.ref.phi.device)

    def spread(self, a):
        return a.expand(a.shape[:-3] + self.shape)

    def charge(self):
        return self.ref.charge() * float(self.times)

    def fields(self, w, precision):
        out = {"phi": self.spread(self.ref.phi), "n": self.spread(self.ref.n)}
        if w.flow and precision == "fp32":
            out["u"] = self.spread(self.ref.moments(self.ref.fluxes()[1])[2])
        elif w.flow:
            out["f"] = self.spread(torch.where(self.ref.fluid, self.ref.gathered(), 0.0))
        return out


class _Gradient:
    """Charge after T steps with the solvent at rest and its gradient, from
    the continuous reading of the occupancy chi in [0, 1] (link factor
    1 + (chi - chi')^2, ion links open by (1 - chi)(1 - chi'), the Poisson row
    (1 - chi)(lap phi + 4 pi l_B rho) + chi (psi - phi)), each step
    differentiated by torch and each solve through its own operator."""

    def __init__(self, w):
        self.w = w
        self.ref = _Reference(w, w.ids, _bulk(w))
        self.dev = self.ref.phi.device

    def charges(self, phi, chi, which):
        w = self.w
        q = torch.zeros_like(phi)
        for i, c in enumerate(_C[1:], 1):
            base = self.ref.inside[i].double() * (1 / 3 if sum(map(abs, c)) == 1 else 1 / 6)
            cj = _at(chi, c)
            q = q + chi * (1.0 - cj) * base * (1.0 + (chi - cj) ** 2) * (_at(phi, c) - phi)
        q = -q / (4.0 * math.pi * w.bjerrum)
        return torch.stack([q[which == e].sum() for e in range(1, w.n_elec + 1)])

    def row(self, phi, n, psi, chi, which):
        w = self.w
        lap = torch.zeros_like(phi)
        for i, c in enumerate(_C[1:], 1):
            base = self.ref.inside[i].double() * (1 / 3 if sum(map(abs, c)) == 1 else 1 / 6)
            lap = lap + base * (1.0 + (chi - _at(chi, c)) ** 2) * (_at(phi, c) - phi)
        rho = n[0] * w.z[0] + n[1] * w.z[1]
        return (1.0 - chi) * (lap + 4.0 * math.pi * w.bjerrum * rho) + chi * (psi[which - 1] - phi)

    def flux(self, n, phi, D, chi):
        out = []
        for k, z in enumerate(self.w.z):
            v = n[k]
            for c in _C[1:]:
                length = math.sqrt(sum(map(abs, c)))
                mu = z * (_at(phi, c) - phi - sum(e * a for e, a in zip(self.w.e_app, c)))
                n1 = _at(n[k], c)
                v = v + (1.0 - chi) * (1.0 - _at(chi, c)) * (D[k] / _A0) / length * 0.5 * (
                    1.0 + torch.exp(-mu)) * ((n1 - n[k]) + n1 * torch.expm1(mu))
            out.append(v)
        return torch.stack(out)

    def back_through_solve(self, phi, n, psi, chi, which, phibar):
        """Adds the solve's part: mu with J^T mu = -phibar, J = d row / d phi."""
        fl = self.ref.fluid
        # fluid rows hold lap, solid rows -1: solid columns see 2 w mu of their fluid neighbours
        mu = self.ref.inverse(torch.where(fl, phibar, 0.0))
        for _ in range(2):
            mu = mu + self.ref.inverse(torch.where(fl, phibar, 0.0) - self.ref.minus_lap(mu))
        from_fluid = torch.zeros_like(mu)
        for i, c in enumerate(_C[1:], 1):
            from_fluid += torch.where(_at(fl, c), self.ref.lap_w[i] * _at(mu, c), 0.0)
        mu = torch.where(fl, mu, phibar + from_fluid)
        args = [a.detach().requires_grad_() for a in (n, psi, chi)]
        r = self.row(phi, args[0], args[1], args[2], which)
        return torch.autograd.grad((r * mu).sum(), args)

    def run(self):
        w, ref = self.w, self.ref
        chi = (~ref.fluid).double()
        which = torch.where(ref.ids == 0, 1, ref.ids)  # fluid nodes would join electrode 1
        psi = torch.tensor(w.psi, dtype=torch.float64, device=self.dev)
        D = torch.tensor(w.D, dtype=torch.float64, device=self.dev)
        states = [(ref.n, ref.phi)]
        for _ in range(w.steps):
            ref.n = torch.where(ref.fluid, ref.fluxes()[0], 0.0)
            ref.solve()
            states.append((ref.n, ref.phi))
        n, phi = states[-1]
        a_phi, a_chi = phi.clone().requires_grad_(), chi.clone().requires_grad_()
        q = self.charges(a_phi, a_chi, which)
        phibar, chibar = torch.autograd.grad(q[0], (a_phi, a_chi))
        nbar, psibar, Dbar = torch.zeros_like(n), torch.zeros_like(psi), torch.zeros_like(D)
        for t in range(w.steps, -1, -1):
            n, phi = states[t]
            gn, gp, gc = self.back_through_solve(phi, n, psi, chi, which, phibar)
            nbar, psibar, chibar = nbar + gn, psibar + gp, chibar + gc
            nbar = torch.where(ref.fluid, nbar, 0.0) if t == w.steps else nbar
            if t == 0:
                break
            n, phi = states[t - 1]
            args = [a.detach().clone().requires_grad_() for a in (n, phi, D, chi)]
            nbar, phibar, gD, gc = torch.autograd.grad((self.flux(*args) * nbar).sum(), args)
            Dbar, chibar = Dbar + gD, chibar + gc
            nbar = torch.where(ref.fluid, nbar, 0.0)
        nbar = torch.where(ref.fluid, nbar, 0.0)
        rho = _bulk(w)[0]
        chibar = chibar - rho * nbar.sum(0)
        return q.detach(), psibar, nbar.sum(), Dbar, chibar


def exact(case, seed):
    c = case
    kind = c["kind"]
    if kind == "batch":
        phi, n, q = [], [], []
        for w in _batch_inputs(c, seed):
            r = _Repeated(w, "plates" if "plates" in w.name else "coax")
            for _ in range(c["steps"]):
                r.ref.step()
            phi.append(r.spread(r.ref.phi).reshape(-1))
            n.append(r.spread(r.ref.n).reshape(-1))
            q.append(torch.cat([r.charge(), r.ref.phi.new_zeros(lbe.LBE_BATCH_MAX_ELECTRODES - w.n_elec)]))
        return {"charge": torch.stack(q), "phi": torch.cat(phi), "n": torch.cat(n)}
    if kind == "gradient":
        ids, psi, debye, D = _gradient_inputs(c, seed)
        w = workloads.Workload("porous", ids, 2, (1, 1, 0), tuple(float(v) for v in psi), _L_B, float(debye),
                               D=tuple(float(v) for v in D), flow=False, steps=c["steps"])
        q, dpsi, drho, dD, dchi = _Gradient(w).run()
        theta = torch.cat([dpsi, (drho * (-2.0 * _bulk(w)[0] / w.debye)).reshape(1), dD])
        return {"charge": q, "theta": theta, "chi": dchi.reshape(-1) if c["slots"] else dchi}
    w, n = _workload(c, seed)
    r = _Repeated(w, c["geometry"], n)
    for _ in range(0 if c.get("restart") else _WARM):
        r.ref.step()
    if kind == "drive":
        q = []
        for psi in _drive(w, c["steps"], seed):
            r.ref.set_voltage(psi)
            r.ref.step()
            q.append(r.charge())
        return {"charge": torch.stack(q), **r.fields(w, c["precision"])}
    if kind == "steps":
        for _ in range(c["steps"]):
            r.ref.step()
        return {"charge": r.charge(), **r.fields(w, c["precision"])}
    f = torch.where(r.ref.fluid, r.ref.gathered(), 0.0)
    q = r.charge()
    return {**r.fields(w, "fp32"), "rho": r.spread(f.sum(0)), "f": r.spread(f),
            "qnode": r.spread(r.ref.charge_map()), "charge": q, "charge_static": q}
