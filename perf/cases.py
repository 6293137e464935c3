"""Measured workloads: what a program built on this package has it do, through its public calls.

Every case is one of these kinds of use:
  point      single-point energies and forces of independent snapshots (data labelling, scans):
             set_state, eam_forces, get, per snapshot;
  md         a stretch of molecular dynamics of one system through step_io: the state in, n steps
             with every list rebuild that falls due, the state and the energies out;
  replicas   the same for a batch of independent replicas in one context, in NVE or with one
             Nose-Hoover thermostat each;
  surrogate  molecular dynamics on the learned per-atom energy;
  training   loss and parameter gradient of the learned energy on a minibatch of frames.
Crystals carry Gaussian displacements and Maxwell-Boltzmann velocities, so that atoms move, lists
are rebuilt and table rows are read as in a running simulation.

Outputs keep the type of the path's arithmetic: float64 for the FP64 and double-float paths; float32
for the mixed path, whose forces are FP32 sums (positions and velocities as a trajectory frame
holds them); float16 for the forces of the bf16 network, whose inputs and activations carry 8
significant bits, so that one of them rounding the other way moves a force by more than an FP32 ulp.
`exact` restates each path in 64-bit torch: all pairs inside the cutoff from a plain cell grid,
the potential from its definition, the integrators step by step.
"""
from __future__ import annotations

import math
import os

import numpy as np
import torch

from paper_1107_2619_gb300 import inputs as I
from paper_1107_2619_gb300 import md

WEIGHTS = os.path.join(os.path.dirname(os.path.abspath(I.__file__)), "data", "surrogate_fe.npz")


def listed():
    return [
        # the smallest call: labelling snapshots of a 432-atom cell, latency and launches only
        {"name": "fe432_point_fp64", "kind": "point", "lattice": "fe", "nx": 6, "ny": 6, "nz": 6,
         "precision": "fp64", "walk": "auto", "tune": False, "temperature": 300.0, "snapshots": 2},
        # the paper's benchmark system: 2,000 atoms of bcc Fe, 1 fs steps, everything at its default
        {"name": "fe2k_md_fp64", "kind": "md", "lattice": "fe", "nx": 10, "ny": 10, "nz": 10,
         "precision": "fp64", "walk": "auto", "tune": False, "temperature": 300.0, "steps": 100,
         "integrator": "verlet", "buffers": "device"},
        # the benchmark's headline: 500,000 atoms of fcc Cu in FP64 over the half list, lanes tuned
        {"name": "cu500k_md_fp64_half", "kind": "md", "lattice": "cu", "nx": 50, "ny": 50, "nz": 50,
         "precision": "fp64", "walk": "half", "tune": True, "temperature": 300.0, "steps": 20,
         "integrator": "verlet", "buffers": "device"},
        # FP64 as a caller gets it who sets nothing (full list, default lanes), an uneven box
        {"name": "cu_uneven_md_fp64", "kind": "md", "lattice": "cu", "nx": 23, "ny": 31, "nz": 29,
         "precision": "fp64", "walk": "auto", "tune": False, "temperature": 600.0, "steps": 10,
         "integrator": "verlet", "buffers": "device"},
        # mixed precision at the headline's size, lanes tuned
        {"name": "cu500k_md_mixed", "kind": "md", "lattice": "cu", "nx": 50, "ny": 50, "nz": 50,
         "precision": "mixed", "walk": "auto", "tune": True, "temperature": 300.0, "steps": 20,
         "integrator": "verlet", "buffers": "device"},
        # double-float precision, an uneven box
        {"name": "cu_uneven_md_df", "kind": "md", "lattice": "cu", "nx": 33, "ny": 27, "nz": 25,
         "precision": "df", "walk": "auto", "tune": True, "temperature": 300.0, "steps": 10,
         "integrator": "verlet", "buffers": "device"},
        # a state kept in the caller's pinned host memory, one step per call (the end-to-end form)
        {"name": "cu500k_step_pinned_fp64", "kind": "md", "lattice": "cu", "nx": 50, "ny": 50, "nz": 50,
         "precision": "fp64", "walk": "half", "tune": True, "temperature": 300.0, "steps": 1,
         "integrator": "verlet", "buffers": "pinned"},
        # two species under the strain ramp: Fe with 0.1 % C
        {"name": "fec250k_strain_mixed", "kind": "md", "lattice": "fec", "nx": 50, "ny": 50, "nz": 50,
         "precision": "mixed", "walk": "auto", "tune": True, "temperature": 600.0, "steps": 20,
         "integrator": "verlet", "buffers": "device"},
        # uneven replicas in one context, NVE, replayed as a graph
        {"name": "fe_replicas32_mixed", "kind": "replicas", "replicas": 32, "low": 10, "high": 30,
         "precision": "mixed", "tune": True, "steps": 20, "thermostat": False},
        # smaller replicas, each under its own thermostat
        {"name": "fe_replicas24_nvt_mixed", "kind": "replicas", "replicas": 24, "low": 8, "high": 20,
         "precision": "mixed", "tune": True, "steps": 20, "thermostat": True},
        # the learned energy's tensor-core network driving half a million atoms
        {"name": "fe524k_surrogate_bf16", "kind": "surrogate", "nx": 64, "ny": 64, "nz": 64, "net": "bf16",
         "temperature": 600.0, "steps": 5},
        # one training minibatch: 16 frames of 2,000 atoms, energies and forces
        {"name": "fe_train_16x2000", "kind": "training", "replicas": 16, "n": 10, "temperature": 600.0},
    ]


def draw(rng):
    def log_int(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    def edges(lo, hi):   # three edges around one logarithmic size
        m = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        return [min(hi, max(lo, int(round(m * rng.uniform(0.85, 1.18))))) for _ in range(3)]

    kind = rng.choice(["point", "md", "md", "md", "replicas", "surrogate", "training"])
    t = float(rng.choice([200.0, 300.0, 450.0, 600.0, 900.0]))
    if kind == "point":
        lat = rng.choice(["fe", "cu"])
        nx, ny, nz = edges(6, 48) if lat == "fe" else edges(7, 34)
        prec = rng.choice(["fp64", "mixed"] + (["df"] if lat == "cu" else []))
        return {"kind": "point", "lattice": lat, "nx": nx, "ny": ny, "nz": nz, "precision": prec, "walk": "auto",
                "tune": False, "temperature": t, "snapshots": rng.choice([1, 2, 3])}
    if kind == "md":
        lat = rng.choice(["fe", "cu", "cu", "fec"])
        nx, ny, nz = edges(7, 46) if lat == "cu" else edges(8, 50)
        prec = rng.choice(["mixed", "fp64", "df"] if lat == "cu" else ["mixed", "fp64"])
        walk = rng.choice(["auto", "half"]) if prec == "fp64" and lat != "fec" else "auto"
        return {"kind": "md", "lattice": lat, "nx": nx, "ny": ny, "nz": nz, "precision": prec, "walk": walk,
                "tune": rng.random() < 0.5, "temperature": t, "steps": log_int(1, 20),
                "integrator": "pc3" if lat != "fec" and rng.random() < 0.2 else "verlet",
                "buffers": rng.choice(["device", "device", "pinned"])}
    if kind == "replicas":
        low = rng.randint(7, 14)
        return {"kind": "replicas", "replicas": log_int(2, 32), "low": low, "high": rng.randint(low, 26),
                "precision": rng.choice(["mixed", "mixed", "fp64"]), "tune": rng.random() < 0.5,
                "steps": log_int(2, 20), "thermostat": rng.random() < 0.5}
    if kind == "surrogate":
        nx, ny, nz = edges(8, 60)
        return {"kind": "surrogate", "nx": nx, "ny": ny, "nz": nz, "net": rng.choice(["bf16", "fp32"]),
                "temperature": t, "steps": log_int(1, 5)}
    return {"kind": "training", "replicas": log_int(2, 16), "n": rng.randint(6, 10), "temperature": t}


# ----------------------------------------------------------------------------- inputs
def _workload(case, seed):
    cells, t, lat = (case["nx"], case["ny"], case["nz"]), case["temperature"], case["lattice"]
    if lat == "fe":
        return I.bcc_fe(0, seed=seed, temperature=t, cells=cells)
    if lat == "cu":
        pos, box = I.replicate(I.FCC_BASIS, cells, 3.615)
        pos = I.gaussian_displace(pos, 0.05, seed)
        pot = I.sc_cu_tables()
        species = np.zeros(len(pos), dtype=np.int32)
        return I.Workload(name="fcc Cu", pos=pos, vel=I.maxwell_boltzmann(pot.masses[species], t, seed),
                          species=species, box=box, potential=pot, skin=0.3, k_max=176, dt_fs=2.0, steps=0, temperature=t)
    fe, box = I.replicate(I.BCC_BASIS, cells, 2.8665)
    sites, _ = I.replicate(I.BCC_OCTA_BASIS, cells, 2.8665)
    n_c = int(round(0.001 * len(fe)))
    chosen = np.sort(np.argsort(I.random_u64(seed, 3, len(sites)), kind="stable")[:n_c])
    species = np.concatenate([np.zeros(len(fe), np.int32), np.ones(n_c, np.int32)])
    pot = I.fe_c_tables()
    return I.Workload(name="bcc Fe-C", pos=I.gaussian_displace(np.concatenate([fe, sites[chosen]]), 0.05, seed),
                      vel=I.maxwell_boltzmann(pot.masses[species], t, seed), species=species, box=box, potential=pot,
                      skin=0.3, k_max=40, dt_fs=1.0, steps=0, temperature=t, strain_rate_zz=-1.0e9)


def _replicas(case, seed):
    m = case["replicas"]
    u = I.random_uniform(seed, 11, 2 * m)
    span = case["high"] - case["low"] + 1
    # the sizes are the case's own (the same for every seed), the temperatures the seed's
    size = case["low"] + np.floor(I.random_uniform(7, 11, m) * span).astype(int)
    temps = 300.0 + 900.0 * u[m:]
    return [I.bcc_fe(int(size[r]), seed=seed + r, temperature=float(temps[r])) for r in range(m)], temps


def _frames(case, seed):
    return [I.bcc_fe(case["n"], seed=seed + 17 * r, temperature=case["temperature"], sigma=0.08)
            for r in range(case["replicas"])]


def _surrogate_workload(case, seed):
    return I.bcc_fe(0, seed=seed, temperature=case["temperature"], cells=(case["nx"], case["ny"], case["nz"]))


def _snapshots(case, w, seed):
    """Independent thermal snapshots of one crystal: each needs its own neighbour list."""
    return [w.pos] + [I.gaussian_displace(w.pos, 0.08, seed + 100 + q) for q in range(1, case["snapshots"])]


def _device(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()


def prepare(case, seed):
    k = case["kind"]
    st = {"case": case}
    if k == "point":
        w = _workload(case, seed)
        s = md.System(w, precision=case["precision"], passes=case["walk"])
        st["snaps"] = [_device(p) for p in _snapshots(case, w, seed)]
        st["force"] = [torch.empty(s.n, 3, dtype=torch.float64, device="cuda") for _ in st["snaps"]]
        st["energy"] = [torch.empty(s.n, dtype=torch.float64, device="cuda") for _ in st["snaps"]]
        s.eam_forces()
    elif k == "md":
        w = _workload(case, seed)
        s = md.System(w, precision=case["precision"], passes=case["walk"], integrator=case["integrator"])
        s.eam_forces()
        if case["tune"]:
            s.tune()
        force = s.forces()
        if case["buffers"] == "pinned":
            pin = lambda a: torch.from_numpy(np.ascontiguousarray(a)).pin_memory().numpy()
            st["in"] = [pin(w.pos), pin(w.vel), pin(force)]
            st["out"] = [pin(np.zeros_like(w.pos)) for _ in range(3)]
        else:
            st["in"] = [_device(w.pos), _device(w.vel), _device(force)]
            st["out"] = [torch.empty_like(st["in"][0]) for _ in range(3)]
    elif k == "replicas":
        ws, temps = _replicas(case, seed)
        s = md.Batch(ws, precision=case["precision"])
        s.eam_forces()
        if case["tune"]:
            s.tune()
        if not case["thermostat"]:
            s.set_graph(True)
        st["temps"] = temps
        st["in"] = [_device(np.concatenate([w.pos for w in ws])), _device(np.concatenate([w.vel for w in ws])),
                    _device(s.forces())]
        st["out"] = [torch.empty_like(st["in"][0]) for _ in range(3)]
    elif k == "surrogate":
        w, d = _surrogate_workload(case, seed), np.load(WEIGHTS)
        s = md.SurrogateSystem(w, d["theta"], d["gmu"], d["ginv"], net=case["net"])
        s.eam_forces()
        st["in"] = [_device(w.pos), _device(w.vel), _device(s.forces())]
        st["out"] = [torch.empty_like(st["in"][0]) for _ in range(3)]
    else:
        ws, d = _frames(case, seed), np.load(WEIGHTS)
        with md.Batch(ws, precision="fp64") as eam:   # the frames' labels
            eam.eam_forces()
            f_ref, e_ref = eam.forces(), np.array([e["pe"] for e in eam.replica_energies()])
        # the weights a training run starts from, with the training set's standardisation
        s = md.SurrogateBatch(ws, I.sur_init_weights(seed), d["gmu"], d["ginv"], net="fp32")
        s.set_reference(e_ref, f_ref)
    st["sys"] = s
    return st


# ----------------------------------------------------------------------------- one pass
def _energies(e, dtype):
    return np.array([e["pe"], e["ke"], e["te"]] + [e["virial"][a][b] for a, b in ((0, 0), (1, 1), (2, 2), (1, 2), (0, 2), (0, 1))],
                    dtype=dtype)


def run(st):
    case, s = st["case"], st["sys"]
    k = case["kind"]
    if k == "point":
        single = torch.float32 if case["precision"] == "mixed" else torch.float64
        pe = []
        for pos, force, energy in zip(st["snaps"], st["force"], st["energy"]):
            s.set_state(pos=pos)
            pe.append(s.eam_forces())
            s.get(md.MD_GET_FORCE, force)
            s.get(md.MD_GET_EATOM, energy)
        return {"pe": np.array(pe, dtype=np.float32 if single == torch.float32 else np.float64),
                "force": [f.to(single) for f in st["force"]], "e_atom": [e.to(single) for e in st["energy"]]}
    if k == "training":
        loss, grad = s.loss_grad(w_e=10.0, w_f=1.0)
        return {"loss": loss.astype(np.float32), "grad": grad}
    if k == "replicas" and case["thermostat"]:
        s.set_thermostat(st["temps"], tau_fs=100.0)   # a stretch starts from zero friction
    e = s.step_io(case["steps"], *st["in"], *st["out"])
    pos, vel, force = st["out"]
    if k == "surrogate":
        half = torch.float16 if case["net"] == "bf16" else torch.float32
        return {"pos": pos.float(), "vel": vel.float(), "force": force.to(half), "energies": np.float32([e["pe"], e["ke"]])}
    if case["precision"] == "mixed":
        if isinstance(pos, np.ndarray):
            return {"pos": pos.astype(np.float32), "vel": vel.astype(np.float32), "force": force.astype(np.float32),
                    "energies": _energies(e, np.float32)}
        return {"pos": pos.float(), "vel": vel.float(), "force": force.float(), "energies": _energies(e, np.float32)}
    return {"pos": pos, "vel": vel, "force": force, "energies": _energies(e, np.float64)}


# ----------------------------------------------------------------------------- work
def _atoms(case):
    if case["kind"] == "replicas":
        span = case["high"] - case["low"] + 1
        size = case["low"] + np.floor(I.random_uniform(7, 11, case["replicas"]) * span).astype(int)
        return int((2 * size ** 3).sum())
    if case["kind"] == "training":
        return case["replicas"] * 2 * case["n"] ** 3
    cells = case["nx"] * case["ny"] * case["nz"]
    lattice = case.get("lattice", "fe")
    return 4 * cells if lattice == "cu" else 2 * cells + (int(round(0.002 * cells)) if lattice == "fec" else 0)


def work(case):
    """Bytes: a list of K entries read by each of the two passes (8 K) and the per-atom state each
    reads and writes once (170 B mixed, 184 B otherwise), per step, and the caller's arrays;
    operations: the pair terms of both passes (47 per list entry; half of them where each pair is
    computed once), or the network's products and the 32 channels of every pair."""
    n, k = _atoms(case), case["kind"]
    if k in ("surrogate", "training"):
        pairs, net = 26 * n, 2 * (32 * 64 + 64 * 64 + 64)
        steps = case.get("steps", 1)
        flops = steps * (pairs * 32 * 2 * 8 + n * net * (2 if k == "surrogate" else 6))
        return {"bytes": steps * n * (2 * 4 * 30 + 3 * 128 + 184) + (144 * n if k == "surrogate" else 24 * n), "flops": flops}
    K = 140 if case.get("lattice") == "cu" else 15
    steps = case["snapshots"] if k == "point" else case["steps"]
    state = 170 if case["precision"] == "mixed" else 184
    half = 0.5 if case.get("walk") == "half" else 1.0
    io = case["snapshots"] * 56 * n if k == "point" else 144 * n
    return {"bytes": steps * n * (8 * K + state) + io, "flops": steps * n * K * 47 * half}


# ----------------------------------------------------------------------------- 64-bit restatement
def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _pairs(pos, box, reach):
    """All i < j (as index pairs) closer than `reach` in the periodic box."""
    n = [max(1, int(float(b) // reach)) for b in box]
    if min(n) < 3:   # a box of few cells: all pairs
        i, j = torch.triu_indices(len(pos), len(pos), 1, device=pos.device)
        d = pos[j] - pos[i]
        d -= box * torch.round(d / box)
        near = (d * d).sum(1) < reach * reach
        return i[near], j[near]
    nc = torch.tensor(n, device=pos.device)
    frac = pos / box
    c = ((frac - torch.floor(frac)) * nc).long().clamp(min=0)
    c = torch.minimum(c, nc - 1)
    cell = (c[:, 2] * n[1] + c[:, 1]) * n[0] + c[:, 0]
    order = torch.argsort(cell, stable=True)
    count = torch.bincount(cell, minlength=n[0] * n[1] * n[2])
    start = torch.cumsum(count, 0) - count
    cap = int(count.max())
    slot = torch.arange(len(pos), device=pos.device) - start[cell[order]]
    table = torch.full((n[0] * n[1] * n[2], cap), -1, dtype=torch.long, device=pos.device)
    table[cell[order], slot] = order
    grid = table.view(n[2], n[1], n[0], cap)
    found = []
    for dz in (0, 1):
        for dy in ((0, 1) if dz == 0 else (-1, 0, 1)):
            for dx in ((0, 1) if dz == dy == 0 else (-1, 0, 1)):
                other = torch.roll(grid, (-dz, -dy, -dx), (0, 1, 2)).reshape(-1, cap)
                step = max(1, (1 << 25) // (cap * cap))
                for c0 in range(0, len(table), step):
                    a, b = table[c0:c0 + step, :, None], other[c0:c0 + step, None, :]
                    live = (a >= 0) & (b >= 0)
                    if dx == dy == dz == 0:
                        live = live & (a < b)
                    i, j = (x[live] for x in torch.broadcast_tensors(a, b))
                    d = pos[j] - pos[i]
                    d -= box * torch.round(d / box)
                    near = (d * d).sum(1) < reach * reach
                    found.append((i[near], j[near]))
    return torch.cat([f[0] for f in found]), torch.cat([f[1] for f in found])


class _Eam:
    """Energies and forces of a potential record in 64 bits."""

    def __init__(self, pot, species):
        self.pot, self.dev = pot, _dev()
        self.sp = torch.from_numpy(np.asarray(species)).long().to(self.dev)
        if pot.kind == I.POT_TABLES:
            ns = pot.n_species
            t = torch.from_numpy(pot.tables).to(self.dev).view(2 * ns * ns + ns, 2, pot.n_knots)
            self.V, self.phi, self.F = t[:ns * ns], t[ns * ns:2 * ns * ns], t[2 * ns * ns:]

    @staticmethod
    def _hermite(tab, which, x, lo, hi):
        nk = tab.shape[2]
        h = (hi - lo) / (nk - 1)
        u = (x - lo) / h
        k = torch.floor(u).clamp(0, nk - 2).long()
        t = u - k
        flat = tab.reshape(-1)
        at = which * (2 * nk) + k
        y0, y1, s0, s1 = flat[at], flat[at + 1], h * flat[at + nk], h * flat[at + nk + 1]
        c2, c3 = 3 * (y1 - y0) - 2 * s0 - s1, 2 * (y0 - y1) + s0 + s1
        y, dy = y0 + t * (s0 + t * (c2 + t * c3)), (s0 + t * (2 * c2 + t * 3 * c3)) / h
        y = torch.where(u < 0, y0 + t * s0, torch.where(u > nk - 1, y1 + (t - 1) * s1, y))
        return y, torch.where(u < 0, s0 / h, torch.where(u > nk - 1, s1 / h, dy))

    def pair_terms(self, i, j, r):
        p = self.pot
        if p.kind == I.POT_FS_ANALYTIC:
            d, c, _, beta, c0, c1, c2 = (float(v) for v in p.fs)
            u, q, dq = r - c, c0 + c1 * r + c2 * r * r, c1 + 2 * c2 * r
            V, dV = torch.where(u < 0, u * u * q, 0.0), torch.where(u < 0, 2 * u * q + u * u * dq, 0.0)
            t = r - d
            f, df = torch.where(t < 0, t * t * (1 + beta / d * t), 0.0), torch.where(t < 0, t * (2 + 3 * beta / d * t), 0.0)
            return V, dV, f, df, f, df
        a, b, ns = self.sp[i], self.sp[j], p.n_species
        V, dV = self._hermite(self.V, a * ns + b, r, p.r_min, p.r_cut)
        f, df = self._hermite(self.phi, a * ns + b, r, p.r_min, p.r_cut)
        if ns == 1:
            return V, dV, f, df, f, df
        return (V, dV, f, df) + self._hermite(self.phi, b * ns + a, r, p.r_min, p.r_cut)

    def __call__(self, pos, box, pairs):
        p = self.pot
        i, j = pairs
        d = pos[j] - pos[i]
        d -= box * torch.round(d / box)
        r2 = (d * d).sum(1)
        keep = r2 < p.r_cut ** 2
        i, j, d, r = i[keep], j[keep], d[keep], torch.sqrt(r2[keep])
        V, dV, fi, dfi, fj, dfj = self.pair_terms(i, j, r)
        rho = torch.zeros(len(pos), dtype=torch.float64, device=pos.device)
        rho.index_add_(0, i, fi)
        rho.index_add_(0, j, fj)
        if p.kind == I.POT_FS_ANALYTIC:
            A = float(p.fs[2])
            F, dF = -A * torch.sqrt(rho), -0.5 * A / torch.sqrt(rho)
        else:
            F, dF = self._hermite(self.F, self.sp, rho, p.rho_min, p.rho_max)
        e = F.clone()
        e.index_add_(0, i, 0.5 * V)
        e.index_add_(0, j, 0.5 * V)
        g = ((dV + dF[i] * dfi + dF[j] * dfj) / r)[:, None] * d
        force = torch.zeros_like(pos)
        force.index_add_(0, i, g)
        force.index_add_(0, j, -g)
        W = -torch.stack([(d[:, a] * g[:, b]).sum() for a, b in ((0, 0), (1, 1), (2, 2), (1, 2), (0, 2), (0, 1))])
        return e, force, W


def _nose(pi, xi, q, gkt, ke, h):
    pi = pi + 0.5 * h * (2 * ke - gkt) / q
    scale = math.exp(-pi * h)
    xi, ke = xi + pi * h, ke * scale * scale
    return pi + 0.5 * h * (2 * ke - gkt) / q, xi, scale


def _trajectory(w, steps, evaluate, reach, integrator="verlet", nvt=None):
    """`steps` steps of one system; evaluate(pos, box, pairs) -> (e per atom, force, W)."""
    dev = _dev()
    put = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).to(dev)
    pos, vel, box = put(w.pos), put(w.vel), put(w.box)
    mass = put(w.potential.masses)[torch.from_numpy(np.asarray(w.species)).long().to(dev)][:, None]
    acc, dt = 1.0 / (I.MVV_TO_EV * mass), w.dt_fs
    s = 1.0 + w.strain_rate_zz * dt * 1.0e-15
    kinetic = lambda v: float((mass * v * v).sum()) * 0.5 * I.MVV_TO_EV
    pairs, at = _pairs(pos, box, reach + 0.9), pos.clone()

    def fresh(x):
        nonlocal pairs, at
        if float(((x - at) ** 2).sum(1).max()) > 0.44 ** 2:
            pairs, at = _pairs(x, box, reach + 0.9), x.clone()
        return evaluate(x, box, pairs)

    e, f, W = evaluate(pos, box, pairs)
    third = torch.zeros_like(pos)
    if nvt:
        gkt = (3 * len(pos) - 3) * I.KB_EV_PER_K * nvt[0]
        q, pi, xi = gkt * nvt[1] ** 2, 0.0, 0.0
    for _ in range(steps):
        if integrator == "pc3":
            a = 0.5 * dt * dt * f * acc
            pos, vel, a1 = pos + dt * vel + a + third, vel + (2 * a + 3 * third) / dt, a + 3 * third
            e, f, W = fresh(pos)
            D = 0.5 * dt * dt * f * acc - a1
            pos, vel, third = pos + D / 6, vel + 5.0 / 6.0 * D / dt, third + D / 3
            continue
        if nvt:
            pi, xi, scale = _nose(pi, xi, q, gkt, kinetic(vel), 0.5 * dt)
            vel = vel * scale
        vel = vel + 0.5 * dt * f * acc
        pos = pos + dt * vel
        if s != 1.0:
            box = box.clone()
            box[2] *= s
            pos[:, 2] *= s
        e, f, W = fresh(pos)
        vel = vel + 0.5 * dt * f * acc
        if nvt:
            pi, xi, scale = _nose(pi, xi, q, gkt, kinetic(vel), 0.5 * dt)
            vel = vel * scale
    pe, ke = float(e.sum()), kinetic(vel)
    return pos, vel, f, np.array([pe, ke, pe + ke] + W.tolist())


class _Net:
    """The learned energy in 64 bits: descriptors, network, forces."""

    def __init__(self, theta=None):
        d, sp = np.load(WEIGHTS), I.SUR_FE
        put = lambda a: torch.from_numpy(np.asarray(a, dtype=np.float32).astype(np.float64)).to(_dev())
        self.theta, self.gmu, self.ginv = put(d["theta"] if theta is None else theta), put(d["gmu"]), put(d["ginv"])
        self.mu = sp["mu0"] + sp["dmu"] * torch.arange(32, dtype=torch.float64, device=_dev())
        self.w2, self.rd = sp["width"] ** 2, sp["rd"]

    def basis(self, r):
        a = r[:, None] - self.mu
        b = torch.exp(-a * a / (2 * self.w2))
        x = math.pi / self.rd * r[:, None]
        fc, dfc = 0.5 * (torch.cos(x) + 1), -0.5 * math.pi / self.rd * torch.sin(x)
        return b * fc, b * (dfc - a / self.w2 * fc)

    def energies(self, G, theta):
        W1, b1, W2, b2, w3, b3 = torch.split(theta, [2048, 64, 4096, 64, 64, 1])
        x = (G - self.gmu) * self.ginv
        a = torch.nn.functional.silu(x @ W1.view(64, 32).T + b1)
        return torch.nn.functional.silu(a @ W2.view(64, 64).T + b2) @ w3 + b3

    def near(self, pos, box, pairs):
        i, j = pairs
        d = pos[j] - pos[i]
        d -= box * torch.round(d / box)
        r2 = (d * d).sum(1)
        k = r2 < self.rd ** 2
        return i[k], j[k], d[k], torch.sqrt(r2[k])

    def descriptors(self, n, i, j, r):
        G = torch.zeros(n, 32, dtype=torch.float64, device=r.device)
        for c in range(0, len(r), 1 << 21):
            b = self.basis(r[c:c + (1 << 21)])[0]
            G.index_add_(0, i[c:c + (1 << 21)], b)
            G.index_add_(0, j[c:c + (1 << 21)], b)
        return G

    def forces(self, g, i, j, d, r):
        force = torch.zeros(len(g), 3, dtype=torch.float64, device=r.device)
        for c in range(0, len(r), 1 << 21):
            s = slice(c, c + (1 << 21))
            p = (((g[i[s]] + g[j[s]]) * self.basis(r[s])[1]).sum(1) / r[s])[:, None] * d[s]
            force = force.index_add(0, i[s], p).index_add(0, j[s], -p)
        return force

    def __call__(self, pos, box, pairs):
        i, j, d, r = self.near(pos, box, pairs)
        G = self.descriptors(len(pos), i, j, r).requires_grad_(True)
        e = self.energies(G, self.theta)
        (g,) = torch.autograd.grad(e.sum(), G)
        return e.detach(), self.forces(g, i, j, d, r), torch.zeros(6, dtype=torch.float64)


def exact(case, seed):
    k = case["kind"]
    if k == "point":
        w = _workload(case, seed)
        eam, box = _Eam(w.potential, w.species), torch.from_numpy(w.box).to(_dev())
        out = {"pe": [], "force": [], "e_atom": []}
        for p in _snapshots(case, w, seed):
            pos = torch.from_numpy(p).to(_dev())
            e, f, _ = eam(pos, box, _pairs(pos, box, w.potential.r_cut))
            for name, v in (("pe", float(e.sum())), ("force", f), ("e_atom", e)):
                out[name].append(v)
        return dict(out, pe=np.array(out["pe"]))
    if k == "md":
        w = _workload(case, seed)
        pos, vel, f, e = _trajectory(w, case["steps"], _Eam(w.potential, w.species), w.potential.r_cut, case["integrator"])
        return {"pos": pos, "vel": vel, "force": f, "energies": e}
    if k == "replicas":
        ws, temps = _replicas(case, seed)
        got = [_trajectory(w, case["steps"], _Eam(w.potential, w.species), w.potential.r_cut,
                           nvt=(float(temps[r]), 100.0) if case["thermostat"] else None) for r, w in enumerate(ws)]
        return {"pos": torch.cat([g[0] for g in got]), "vel": torch.cat([g[1] for g in got]),
                "force": torch.cat([g[2] for g in got]), "energies": np.sum([g[3] for g in got], axis=0)}
    net = _Net(I.sur_init_weights(seed) if k == "training" else None)
    if k == "surrogate":
        pos, vel, f, e = _trajectory(_surrogate_workload(case, seed), case["steps"], net, net.rd)
        return {"pos": pos, "vel": vel, "force": f, "energies": e[:2]}
    theta = net.theta.clone().requires_grad_(True)
    R, N, le, lf = case["replicas"], 2 * case["n"] ** 3, 0.0, 0.0
    for w in _frames(case, seed):
        pos, box = torch.from_numpy(w.pos).to(_dev()), torch.from_numpy(w.box).to(_dev())
        pairs = _pairs(pos, box, net.rd)
        e_ref, f_ref, _ = _Eam(w.potential, w.species)(pos, box, pairs)
        i, j, d, r = net.near(pos, box, pairs)
        G = net.descriptors(N, i, j, r).requires_grad_(True)
        e = net.energies(G, theta)
        (g,) = torch.autograd.grad(e.sum(), G, create_graph=True)
        f = net.forces(g, i, j, d, r)
        le = le + 10.0 / R * ((e.sum() - e_ref.sum()) / N) ** 2
        lf = lf + ((f - f_ref) ** 2).sum() / (3 * N * R)
    (grad,) = torch.autograd.grad(le + lf, theta)
    return {"loss": np.array([float(le.detach()), float(lf.detach())]), "grad": grad}
