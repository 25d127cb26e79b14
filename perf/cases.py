"""What the performance of this framework is measured on: calls that a user's program makes, through
the public binding, with seeded synthetic inputs.

A case is a dict of plain values. ``listed()`` names the fixed ones, ``draw(rng)`` gives others of
the same ranges, ``prepare`` makes what a program holds before the call (contexts with their
particles, networks, input tensors), ``run`` is one pass and returns its results, ``work`` counts
the bytes and operations a pass cannot do without, and ``exact`` is the same pass in plain torch
and numpy in 64 bits.

Kinds of case:

- ``flow``: a suspension advances ``steps`` time steps, then the particle state is read (with
  ``fields`` the density and velocity fields too).
- ``batch``: an ensemble of independent cells advances ``steps`` steps as one batch, then every
  cell's particle state is read.
- ``predict``: closure inputs of every particle from the current state, then the closure network.
- ``train``: the closure network trains ``epochs`` epochs on pairs held on the device.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1105_2904_gb300 import autotune, closure, lbmp
from paper_1105_2904_gb300 import workloads as W

# The benchmark's periodic suspension: spheres r = 8, 25.6 % solid, tau 0.6, body force 1e-6
# on fluid and particles, velocities N(0, 1e-3), density ratio 1.2.
_SUSPENSION = {"kind": "flow", "lattice": "D3Q19", "precision": "fp32", "streaming": "pull", "walls": "", "lid": 0.0,
               "radius": 8.0, "solid": 0.256, "density": 1.2, "tau": 0.6, "force": 1e-6, "gravity": 0.0,
               "sigma": 1e-3, "gap": 1.0, "block": 0, "fields": False}


def _suspension(name, n, steps, **more):
    return dict(_SUSPENSION, name=name, nx=n, ny=n, nz=n, steps=steps, **more)


def listed():
    return [
        # Flow past a fixed disk in a small 2D channel, the parity configuration: 8192 sites in FP64
        # storage, the drag and the fields read every few steps. Launches and latency are all of it.
        {"name": "channel_disk_fp64", "kind": "flow", "lattice": "D2Q9", "precision": "fp64", "streaming": "pull",
         "walls": "", "lid": 0.0, "nx": 128, "ny": 64, "nz": 1, "radius": 8.0, "solid": 0.0, "density": math.inf,
         "tau": 0.8, "force": 1e-6, "gravity": 0.0, "sigma": 0.0, "gap": 1.0, "block": 0, "steps": 10, "fields": True},
        # Hundreds of disks settling in a closed 2D box (1024 x 2048 sites, 500 disks r = 10).
        {"name": "sedimentation_2d", "kind": "flow", "lattice": "D2Q9", "precision": "fp32", "streaming": "pull",
         "walls": "xy", "lid": 0.0, "nx": 1024, "ny": 2048, "nz": 1, "radius": 10.0, "solid": 0.075, "density": 1.5,
         "tau": 0.7, "force": 0.0, "gravity": -1e-5, "sigma": 0.0, "gap": 2.0, "block": 0, "steps": 20,
         "fields": False},
        # The headline: the 512^3 suspension of 16000 spheres in FP32 storage.
        _suspension("suspension_512_fp32", 512, 2, block=128),
        # The same box with half the memory, FP16 scaled deviations.
        _suspension("suspension_512_fp16", 512, 2, precision="fp16", block=128),
        # A 256^3 suspension in BF16 storage, read more often.
        _suspension("suspension_256_bf16", 256, 4, precision="bf16", block=128),
        # The 64^3 replica with the same solid fraction (31 spheres), fields read: many short
        # steps, as in parameter studies and tests.
        _suspension("suspension_64_fp32", 64, 20, fields=True),
        # Odd, ragged sizes: plane Couette flow of a dilute suspension between no-slip walls, one
        # of them moving, in a box no dimension of which divides by two.
        dict(_SUSPENSION, name="couette_odd_fp32", nx=161, ny=93, nz=117, radius=6.0, solid=0.10, tau=0.8, walls="z",
             lid=0.01, steps=8),
        # FP64 storage in 3D, the form that reproduces the oracle bit for bit (validation runs).
        _suspension("suspension_160_fp64", 160, 4, precision="fp64"),
        # One distribution buffer instead of two: the scheme for boxes that would not fit otherwise.
        _suspension("inplace_384_fp32", 384, 2, streaming="inplace", block=128),
        # 64 uneven cells (edges 32-128, 1-8 spheres each) stepped together as one batch.
        {"name": "ensemble_64_fp32", "kind": "batch", "precision": "fp32", "cells": 64, "sizes_seed": 4, "edge_lo": 32,
         "edge_hi": 128, "spheres": 8, "steps": 10},
        # Learned closure in use: inputs of 200 spheres of a coarse 128^3 cell, then the network.
        {"name": "closure_predict_200", "kind": "predict", "n": 128, "spheres": 200, "steps": 40},
        # Learned closure in training: one epoch over the 3072 pairs that 384 small cells give, in
        # minibatches of 128.
        {"name": "closure_train_3072", "kind": "train", "rows": 3072, "batch": 128, "epochs": 1},
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["flow3", "flow3", "flow3", "flow2", "batch", "predict", "train"])
    if kind == "flow3":
        precision = rng.choice(["fp32", "fp32", "fp16", "bf16", "fp64"])
        radius = rng.uniform(4.0, 10.0)
        walls = rng.choice(["", "", "z", "yz"])
        # up to 340^3 sites; FP64 boxes stay below 192^3
        nx, ny, nz = (log(40, 192 if precision == "fp64" else 340) for _ in range(3))
        sites = nx * ny * nz
        return dict(_SUSPENSION, precision=precision, nx=nx, ny=ny, nz=nz, walls=walls,
                    lid=rng.choice([0.0, 0.01]) if walls else 0.0, radius=radius,
                    solid=rng.uniform(0.02, 0.2) if not walls else rng.uniform(0.02, 0.1), tau=rng.uniform(0.55, 1.0),
                    streaming=rng.choice(["pull", "pull", "inplace"]), steps=rng.randint(2, 6),
                    fields=sites < 500_000)
    if kind == "flow2":
        walls = rng.choice(["", "xy", "y"])
        return {"kind": "flow", "lattice": "D2Q9", "precision": rng.choice(["fp32", "fp16", "fp64"]),
                "streaming": "pull", "walls": walls, "lid": 0.0, "nx": log(100, 2048), "ny": log(100, 2048), "nz": 1,
                "radius": rng.uniform(4.0, 12.0), "solid": rng.uniform(0.02, 0.1), "density": 1.5,
                "tau": rng.uniform(0.6, 1.0), "force": 0.0 if walls == "xy" else 1e-6,
                "gravity": -1e-5 if "y" in walls else 0.0, "sigma": 1e-3, "gap": 2.0, "block": 0,
                "steps": rng.randint(5, 20), "fields": False}
    if kind == "batch":
        lo = rng.randint(28, 48)
        return {"kind": "batch", "precision": rng.choice(["fp32", "fp32", "fp16"]), "cells": log(4, 48),
                "sizes_seed": rng.randint(1, 10 ** 6), "edge_lo": lo, "edge_hi": rng.randint(lo + 16, 128), "spheres": rng.randint(1, 8), "steps": rng.randint(4, 10)}
    if kind == "predict":
        n = log(32, 160)
        return {"kind": "predict", "n": n, "spheres": max(2, int(200 * (n / 128.0) ** 3)), "steps": rng.randint(10, 40)}
    return {"kind": "train", "rows": log(256, 4096), "batch": rng.choice([64, 96, 128, 200]), "epochs": 1}


# ---- inputs ----------------------------------------------------------------------------------

def _walls(case):
    return tuple(int(a in case["walls"]) for a in "xyz")


def _flow_particles(case, seed):
    """(centres, radii, densities, velocities) of a flow case. Large periodic boxes repeat a
    randomly filled block (``block`` sites wide) with velocities of their own for every sphere."""
    two_d = case["lattice"] == "D2Q9"
    dims = (case["nx"], case["ny"], case["nz"])
    r = float(case["radius"])
    if case["solid"] == 0.0:  # one particle in the middle
        c = np.array([[dims[0] / 2, dims[1] / 2, 0.0 if two_d else dims[2] / 2]])
        c[0, :2 if two_d else 3] += np.random.default_rng(seed).uniform(-0.5, 0.5, 2 if two_d else 3)
    else:
        b = case["block"] or 0
        box = tuple(b or v for v in dims[:2 if two_d else 3])
        size = math.pi * r * r if two_d else 4.0 / 3.0 * math.pi * r ** 3
        n = max(1, int(round(case["solid"] * math.prod(box) / size)))
        c, _ = W.rsa_centers(box, n, r, seed, case["gap"], _walls(case))
        if b:
            at = np.stack(np.meshgrid(*[np.arange(v // b) * float(b) for v in dims], indexing="ij"), -1).reshape(-1, 1, 3)
            c = (c[None] + at).reshape(-1, 3)
    n = len(c)
    v = np.zeros((n, 3))
    if case["sigma"]:
        v = W.gaussian_velocities(n, case["sigma"], seed + 1, 2 if two_d else 3)
    return c, np.full(n, r), np.full(n, float(case["density"])), v


def _ensemble(case, seed):
    """The cells of a batch case (sizes, spheres and relaxation times belong to the case), each
    shifted as a whole by a random vector, with random velocities."""
    e = W.ensemble_cells(case["cells"], case["sizes_seed"], (case["edge_lo"], case["edge_hi"]), (1, case["spheres"]))
    g = np.random.default_rng(seed)
    for k, d in enumerate(e.dims):
        e.centers[k] = np.mod(e.centers[k] + g.uniform(0.0, d), d)
        e.velocities[k] = g.normal(0.0, 1e-3, size=(len(e.radii[k]), 3))
    return e


def _train_data(case, seed):
    """Closure pairs with the statistics of the real ones: correlated, standardised moments and
    three offsets in [0, 1); targets a smooth function of the inputs with noise."""
    g = np.random.default_rng(seed)
    k, o = closure.SIZES[0], closure.SIZES[-1]
    low = g.normal(size=(case["rows"], 24))
    x = low @ g.normal(size=(24, k)) / math.sqrt(24.0) + 0.2 * g.normal(size=(case["rows"], k))
    x[:, -3:] = g.uniform(0.0, 1.0, size=(case["rows"], 3))
    t = np.tanh(low @ g.normal(size=(24, o)) / math.sqrt(24.0)) + 0.1 * g.normal(size=(case["rows"], o))
    return x.astype(np.float32), t.astype(np.float32), g


def _layers(g):
    out = []
    for a, b in zip(closure.SIZES[:-1], closure.SIZES[1:]):
        bound = math.sqrt(6.0 / a)
        out.append([g.uniform(-bound, bound, size=(b, a)), g.uniform(-0.1, 0.1, size=b)])
    return out


def _predict_setup(case, seed):
    """Fixed spheres r = 3 of a coarse closure cell, and the network with its input scaling."""
    n = case["n"]
    c, r = W.rsa_centers((n, n, n), case["spheres"], 3.0, seed, 2.0)
    g = np.random.default_rng(seed + 1)
    layers = _layers(g)
    shift = 0.1 * g.normal(size=closure.SIZES[0])
    scale = g.uniform(0.5, 2.0, size=closure.SIZES[0])
    return c, r, layers, shift, scale


_PREDICT_TAU, _PREDICT_ACCEL, _PREDICT_U, _SPACING = 1.0, 1e-5, 2e-4, 4.0


def prepare(case, seed):
    if case["kind"] == "flow":
        lattice = lbmp.LBM_D2Q9 if case["lattice"] == "D2Q9" else lbmp.LBM_D3Q19
        sim = lbmp.Simulation(lattice, case["nx"], case["ny"], case["nz"], case["tau"],
                              body_force=(case["force"], 0.0, 0.0), precision=case["precision"], walls=_walls(case),
                              gravity=(0.0, case["gravity"], 0.0), body_force_on_particles=case["force"] != 0.0,
                              wall_velocity={5: (case["lid"], 0.0, 0.0)} if case["lid"] else None,
                              streaming=case["streaming"])
        sim.add_particles(*_flow_particles(case, seed))
        return {"case": case, "sim": sim}
    if case["kind"] == "batch":
        e = _ensemble(case, seed)
        b = lbmp.Batch(lbmp.LBM_D3Q19, e.dims, e.taus, [e.body_force] * len(e.dims), precision=case["precision"],
                       body_force_on_particles=e.body_force_on_particles)
        for k in range(len(e.dims)):
            b.add_particles(k, e.centers[k], e.radii[k], e.densities[k], e.velocities[k])
        b.set_tuning(tile_width=autotune.width_policies(b.dims)["min_waste"], steps_per_graph=case["steps"])
        return {"case": case, "batch": b}
    if case["kind"] == "predict":
        n = case["n"]
        c, r, layers, shift, scale = _predict_setup(case, seed)
        sim = lbmp.Simulation(lbmp.LBM_D3Q19, n, n, n, _PREDICT_TAU, body_force=(_PREDICT_ACCEL, 0.0, 0.0))
        sim.add_particles(c, r, np.full(len(r), math.inf))
        sim.step(case["steps"])
        net = lbmp.MLP(closure.SIZES)
        net.set_params(layers)
        net.set_input_scaling(shift, scale)
        return {"case": case, "sim": sim, "net": net}
    x, t, g = _train_data(case, seed)
    net = lbmp.MLP(closure.SIZES)
    net.set_params(_layers(g))
    net.set_input_scaling(x.mean(0), 1.0 / np.maximum(x.std(0), 1e-6))
    return {"case": case, "net": net, "x": torch.tensor(x, device="cuda"), "t": torch.tensor(t, device="cuda")}


def run(state):
    case = state["case"]
    if case["kind"] == "flow":
        sim = state["sim"]
        sim.step(case["steps"])
        out = dict(sim.get_particles())
        if case["fields"]:
            out["rho"], out["velocity"] = sim.get_fields()
        return out
    if case["kind"] == "batch":
        b = state["batch"]
        b.step(case["steps"])
        cells = [b.cell(k).get_particles() for k in range(len(b))]
        return {k: np.concatenate([c[k] for c in cells]) for k in ("x", "u", "omega", "force", "torque")}
    if case["kind"] == "predict":
        x = state["sim"].closure_features(closure.N_SIDE, _SPACING, _PREDICT_U)
        return {"inputs": x, "correction": state["net"].forward(x)}
    net = state["net"]
    loss = net.train(state["x"], state["t"], batch=case["batch"], epochs=case["epochs"], lr=5e-4, seed=1)
    return {"loss": loss, "params": net.params()}


def work(case):
    """A time step reads and writes every population once (2 Q values a site); about 12 Q
    operations a site. The network's products are 2 rows in out, three times that in training."""
    size = {"fp64": 8, "fp32": 4, "fp16": 2, "bf16": 2}
    mlp = sum(a * b for a, b in zip(closure.SIZES[:-1], closure.SIZES[1:]))
    if case["kind"] == "flow":
        q = 9 if case["lattice"] == "D2Q9" else 19
        sites = case["nx"] * case["ny"] * case["nz"]
        bytes_ = 2.0 * q * size[case["precision"]] * sites * case["steps"]
        if case["fields"]:
            bytes_ += sites * (q * size[case["precision"]] + 32.0)
        return {"bytes": bytes_, "flops": 12.0 * q * sites * case["steps"]}
    if case["kind"] == "batch":
        sites = case["cells"] * ((case["edge_lo"] + case["edge_hi"]) / 2.0) ** 3
        return {"bytes": 2.0 * 19 * size[case["precision"]] * sites * case["steps"],
                "flops": 12.0 * 19 * sites * case["steps"]}
    if case["kind"] == "predict":
        n, k = case["spheres"], closure.SIZES[0]
        nodes = n * closure.N_SIDE ** 3
        return {"bytes": nodes * 8.0 * 19 * 4 + n * (2.0 * k + 6) * 4 + 2.0 * mlp, "flops": 2.0 * n * mlp + nodes * 8.0 * 100}
    rows = case["rows"] // min(case["batch"], case["rows"]) * min(case["batch"], case["rows"]) * case["epochs"]
    steps = rows // min(case["batch"], case["rows"])
    return {"bytes": 4.0 * rows * (closure.SIZES[0] + 6) + 28.0 * mlp * steps, "flops": 6.0 * rows * mlp}


# ---- the same in 64 bits -----------------------------------------------------------------------

# populations of one box that are still advanced in 64 bits
_EXACT_VALUES = 2_600_000_000 if torch.cuda.is_available() else 100_000_000


def exact(case, seed):
    if case["kind"] == "flow":
        if case["nx"] * case["ny"] * case["nz"] * (9 if case["lattice"] == "D2Q9" else 19) > _EXACT_VALUES:
            return None
        c, r, d, v = _flow_particles(case, seed)
        s = _Plain(case["lattice"] == "D2Q9", (case["nx"], case["ny"], case["nz"]), case["tau"], case["force"],
                   _walls(case), case["gravity"], case["lid"], case["force"] != 0.0, c, r, d, v)
        s.step(case["steps"])
        out = s.particles()
        if case["fields"]:
            rho, u = s.fields()
            out["rho"], out["velocity"] = rho.cpu().numpy(), u.cpu().numpy()
        return out
    if case["kind"] == "batch":
        e = _ensemble(case, seed)
        cells = []
        for k in range(len(e.dims)):
            s = _Plain(False, e.dims[k], e.taus[k], e.body_force[0], (0, 0, 0), 0.0, 0.0, True, e.centers[k],
                       e.radii[k], e.densities[k], e.velocities[k])
            s.step(case["steps"])
            cells.append(s.particles())
        return {k: np.concatenate([c[k] for c in cells]) for k in ("x", "u", "omega", "force", "torque")}
    if case["kind"] == "predict":
        n = case["n"]
        c, r, layers, shift, scale = _predict_setup(case, seed)
        s = _Plain(False, (n, n, n), _PREDICT_TAU, _PREDICT_ACCEL, (0, 0, 0), 0.0, 0.0, False, c, r,
                   np.full(len(r), math.inf), np.zeros((len(r), 3)))
        s.step(case["steps"])
        rho, u = s.fields()
        m = torch.cat([rho[..., None] - 1.0, u], -1).cpu().numpy()
        side = closure.N_SIDE
        node = _SPACING * (np.arange(side) - 0.5 * (side - 1))
        kk, jj, ii = np.meshgrid(node, node, node, indexing="ij")
        pos = c[:, None, :] + np.stack([ii, jj, kk], -1).reshape(1, -1, 3)
        lo = np.floor(pos).astype(np.int64)
        w = pos - lo
        acc = np.zeros(pos.shape[:2] + (4,))
        for corner in range(8):
            hi = np.array([corner & 1, corner >> 1 & 1, corner >> 2 & 1])
            at = (lo + hi) % n
            acc += np.prod(np.where(hi, w, 1.0 - w), -1)[..., None] * m[at[..., 2], at[..., 1], at[..., 0]]
        x = np.concatenate([(acc / _PREDICT_U).reshape(len(c), -1), c - np.floor(c)], 1)
        h = (x - shift) * scale
        for k, (wt, b) in enumerate(layers):
            h = h @ wt.T + b
            if k + 1 < len(layers):
                h = np.maximum(h, 0.0)
        return {"inputs": x, "correction": h}
    return None  # the minibatches' order is the library's own


class _Plain:
    """The method in plain torch, 64 bits: collision, momentum transfer at boundary sites,
    rigid-body update with contacts, imposition at internal sites, propagation."""

    def __init__(self, two_d, dims, tau, force, walls, gravity, lid, force_on_particles, c, r, density, v):
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        D = 2 if two_d else 3
        self.D, self.dims, self.tau, self.walls, self.lid = D, tuple(int(a) for a in dims), tau, walls, lid
        vel = [(x, y, z) for z in ((0,) if two_d else (-1, 0, 1)) for y in (-1, 0, 1) for x in (-1, 0, 1)
               if abs(x) + abs(y) + abs(z) <= 2]
        w2 = {0: 4 / 9, 1: 1 / 9, 2: 1 / 36} if two_d else {0: 1 / 3, 1: 1 / 18, 2: 1 / 36}
        self.c, self.w = vel, [w2[abs(x) + abs(y) + abs(z)] for x, y, z in vel]
        self.opp = [vel.index((-x, -y, -z)) for x, y, z in vel]
        nx, ny, nz = self.dims
        self.N = nx * ny * nz
        self.F = np.array([force, 0.0, 0.0])
        self.f = torch.tensor(self.w, dtype=torch.float64, device=self.dev)[:, None].repeat(1, self.N)
        # particles
        n = len(c)
        self.x0 = np.array(c, dtype=np.float64).reshape(n, 3)
        self.x, self.r = self.x0.copy(), np.asarray(r, dtype=np.float64)
        self.A = np.floor(self.x0).astype(np.int64)
        self.phi, self.K = self.x0 - self.A, self.A.copy()
        self.u, self.om = np.array(v, dtype=np.float64).reshape(n, 3), np.zeros((n, 3))
        rho = np.asarray(density, dtype=np.float64)
        vol = math.pi * self.r ** 2 if two_d else 4.0 / 3.0 * math.pi * self.r ** 3
        self.inv_m = 1.0 / (rho * vol)
        self.inv_I = self.inv_m / ((0.5 if two_d else 0.4) * self.r ** 2)
        self.ext = np.zeros((n, 3))
        self.ext[:, 1] += gravity * (1.0 - 1.0 / rho)
        if force_on_particles:
            self.ext += self.F / rho[:, None]
        self.ext[np.isinf(rho)] = 0.0
        self.force, self.torque = np.zeros((n, 3)), np.zeros((n, 3))
        # sites of each particle about floor(x0): offsets and class (0 internal, 1 boundary, 2 inside)
        m = int(math.ceil(self.r.max())) + 2
        ax = torch.arange(-m, m + 1, device=self.dev)
        o = torch.stack(torch.meshgrid(ax, ax, ax if D == 3 else ax[m:m + 1], indexing="ij"), -1)
        pid, off, cls = [], [], []
        for p in range(0, n, 256):
            d = o - torch.tensor(self.phi[p:p + 256], device=self.dev)[:, None, None, None]
            inside = (d * d).sum(-1) <= torch.tensor(self.r[p:p + 256] ** 2, device=self.dev)[:, None, None, None]
            bs = inside & self._near(~inside)
            is_ = inside & ~bs & self._near(bs)
            at = inside.nonzero()
            pid.append(at[:, 0] + p)
            off.append(o[at[:, 1], at[:, 2], at[:, 3]])
            cls.append(torch.where(is_, 0, torch.where(bs, 1, 2))[inside])
        self.e_pid, self.e_off, self.e_cls = torch.cat(pid), torch.cat(off), torch.cat(cls)
        self._own()

    def _near(self, m):
        """Sites with a neighbour in m, per particle (periodic roll; the margin is empty)."""
        out = torch.zeros_like(m)
        for c in self.c:
            if any(c):
                out |= torch.roll(m, c, (1, 2, 3))
        return out

    def _own(self):
        """Owner map: at a contested site the lowest (class, particle) wins."""
        K = torch.tensor(self.K, device=self.dev)
        at = K[self.e_pid] + self.e_off
        ok = torch.ones(len(at), dtype=torch.bool, device=self.dev)
        for k in range(3):
            n = self.dims[k]
            if self.walls[k] and k < self.D:
                ok &= (at[:, k] >= 0) & (at[:, k] < n)
            at[:, k] %= n
        site = (at[:, 2] * self.dims[1] + at[:, 1]) * self.dims[0] + at[:, 0]
        code = self.e_cls * (1 << 30) + self.e_pid
        best = torch.full((self.N,), 1 << 40, dtype=torch.int64, device=self.dev)
        best.scatter_reduce_(0, site[ok], code[ok], "amin")
        own = ok & (best[site] == code)
        self.sites = [(site[own & (self.e_cls == k)], self.e_pid[own & (self.e_cls == k)],
                       self.e_off[own & (self.e_cls == k)]) for k in (0, 1)]

    def _feq(self, i, rho, u):
        cu = sum(self.c[i][k] * u[k] for k in range(3))
        return self.w[i] * rho * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * (u[0] * u[0] + u[1] * u[1] + u[2] * u[2]))

    def _moments(self, f):
        rho = f.sum(0)
        j = [sum(self.c[i][k] * f[i] for i in range(len(self.c)) if self.c[i][k]) if k < self.D else torch.zeros_like(rho)
             for k in range(3)]
        return rho, j

    def _rigid(self, pid, off):
        r = off.double() - torch.tensor(self.phi, device=self.dev)[pid]
        u = torch.tensor(self.u, device=self.dev)[pid]
        om = torch.tensor(self.om, device=self.dev)[pid]
        return r, u + torch.linalg.cross(om, r)

    def _min(self, d, k):
        n = self.dims[k]
        return d if self.walls[k] or k >= self.D else d - n * np.floor(d / n + 0.5)

    def step(self, steps):
        for _ in range(steps):
            self._step()

    def _step(self):
        f, F, om = self.f, self.F, 1.0 / self.tau
        rho, j = self._moments(f)
        u = [(j[k] + 0.5 * F[k]) / rho for k in range(3)]
        uF = sum(u[k] * F[k] for k in range(3))
        for i, c in enumerate(self.c):
            cu, cF = sum(c[k] * u[k] for k in range(3)), float(np.dot(c, F))
            f[i] += om * (self._feq(i, rho, u) - f[i]) + (1.0 - 0.5 * om) * self.w[i] * (3.0 * (cF - uF) + 9.0 * cu * cF)
        # momentum transfer at the boundary sites
        n = len(self.x)
        site, pid, off = self.sites[1]
        r, up = self._rigid(pid, off)
        fb = f[:, site]
        rho, j = self._moments(fb)
        dp = rho[:, None] * up - torch.stack(j, -1)
        for i in range(len(self.c)):
            f[i, site] = self._feq(i, rho, up.T)
        tot = torch.zeros(n, 6, dtype=torch.float64, device=self.dev)
        tot.index_add_(0, pid, torch.cat([dp, torch.linalg.cross(r, dp)], 1))
        tot = tot.cpu().numpy()
        self.force, self.torque = -tot[:, :3], -tot[:, 3:]
        un = self.u - tot[:, :3] * self.inv_m[:, None] + self.ext
        self.om = self.om - tot[:, 3:] * self.inv_I[:, None]
        self._contacts(un)
        for k in range(self.D):
            if self.walls[k]:
                xp = self.x[:, k] + un[:, k]
                lo, hi = xp + 0.5 < self.r, (self.dims[k] - 0.5) - xp < self.r
                flip = ((lo & (un[:, k] < 0)) | (~(lo & (un[:, k] < 0)) & hi & (un[:, k] > 0))) & (self.inv_m != 0.0)
                un[flip, k] *= -1.0
        self.u = un
        self.x[:, :self.D] += un[:, :self.D]
        K = self.A + np.floor(self.x - self.x0 + 0.5).astype(np.int64)
        if (K != self.K).any():
            self.K = K
            self._own()
        # imposition at the internal sites
        site, pid, off = self.sites[0]
        _, up = self._rigid(pid, off)
        rho = f[:, site].sum(0)
        for i in range(len(self.c)):
            f[i, site] = self._feq(i, rho, up.T)
        self._stream()

    def _contacts(self, un):
        n = len(self.x)
        if n < 2:
            return
        xp, r = torch.tensor(self.x + un, device=self.dev), torch.tensor(self.r, device=self.dev)
        cand = []
        for i in range(0, n, 1024):
            d2 = 0.0
            for k in range(self.D):
                d = xp[None, :, k] - xp[i:i + 1024, None, k]
                if not self.walls[k]:
                    d = d - self.dims[k] * torch.floor(d / self.dims[k] + 0.5)
                d2 = d2 + d * d
            hit = (d2 < (r[None] + r[i:i + 1024, None]) ** 2).nonzero() + torch.tensor([i, 0], device=self.dev)
            cand += [(int(a), int(b)) for a, b in hit.cpu().numpy() if a < b]
        for i, j in cand:
            den = self.inv_m[i] + self.inv_m[j]
            d = np.array([self._min(self.x[j, k] - self.x[i, k], k) for k in range(3)])
            dn = math.sqrt(float(d @ d))
            if den == 0.0 or dn == 0.0:
                continue
            w = float((un[j] - un[i]) @ d) / dn
            if w < 0.0:
                un[i] += 2.0 * self.inv_m[i] * w / den * d / dn
                un[j] -= 2.0 * self.inv_m[j] * w / den * d / dn

    def _stream(self):
        nx, ny, nz = self.dims
        f = self.f.view(-1, nz, ny, nx)
        out = torch.empty_like(f)
        for i, c in enumerate(self.c):
            out[i] = torch.roll(f[i], (c[2], c[1], c[0]), (0, 1, 2))
        for i, c in enumerate(self.c):  # moves that leave through a wall bounce back where they started
            face = torch.full((nz, ny, nx), -1, dtype=torch.int64, device=self.dev)
            for k in (2, 1, 0):
                if self.walls[k] and c[k]:
                    last = 0 if c[k] < 0 else self.dims[k] - 1
                    face.select(2 - k, last).fill_(2 * k + (c[k] > 0))
            hit = face >= 0
            if any(self.walls[k] and c[k] for k in range(3)):
                back = f[i][hit]
                if self.lid:
                    back = back - (face[hit] == 5).double() * (6.0 * self.w[i] * c[0] * self.lid)
                out[self.opp[i]][hit] = back
        self.f = out.view(len(self.c), -1)

    def particles(self):
        return {"x": self.x.copy(), "u": self.u.copy(), "omega": self.om.copy(), "force": self.force.copy(),
                "torque": self.torque.copy()}

    def fields(self):
        rho, j = self._moments(self.f)
        u = torch.stack([(j[k] + 0.5 * self.F[k]) / rho for k in range(3)], -1)
        nx, ny, nz = self.dims
        return rho.view(nz, ny, nx), u.view(nz, ny, nx, 3)
