"""The work a user of the engine has it do, as timed cases.

A case is a dict: "kind" names the path, the other entries its sizes and
options.  prepare() makes what a program holds before the call (contexts,
meshes, densities, charges), run() makes the call through the public binding
(paper_2110_09214_gb300.obem), exact() states the result in 64 bits with torch
alone.  Workloads are those of inputs.py: parallel plates, the avalanche
counter, the single and the double GEM, the batched sweep.
"""
import functools
import math

import numpy as np
import torch

from paper_2110_09214_gb300 import inputs, obem

KC = 1.0 / (4.0 * math.pi * 8.8541878128e-12)
EPS0 = 8.8541878128e-12
DEV = "cuda" if torch.cuda.is_available() else "cpu"
F64 = dict(dtype=torch.float64, device=DEV)
PRECISION = {"fp32": obem.OBEM_LU_FP32, "tf32": obem.OBEM_LU_TF32, "bf16": obem.OBEM_LU_BF16}
EXACT_CELLS = 13000       # largest dense system that exact() solves in 64 bits
EXACT_PAIRS = 1.5e11      # most charge pairs that exact() sums in 64 bits


def listed():
    return [
        # The first program a user writes: 1000 electrons in a Maxwell-model gas
        # between two plates of 1024 cells, a few tracking steps in a row.
        {"name": "steps_plates", "kind": "steps", "mesh": "plates", "cells": 1024, "n": 1000, "gas": "maxwell",
         "steps": 4, "groups": False},
        # Early avalanche in the plate counter: 1e4 charges, 4096 cells, argon-like gas.
        {"name": "step_avalanche", "kind": "steps", "mesh": "plates", "cells": 4096, "n": 10_000, "gas": "argon",
         "steps": 1, "groups": False},
        # One fused step of a GEM hole's avalanche with the full 60k-cell mesh.
        {"name": "step_gem", "kind": "steps", "mesh": "gem", "cells": 60_000, "n": 100_000, "gas": "argon",
         "steps": 1, "groups": True},
        # The tracking part at full size, the field given by the caller (a user's own field solver).
        {"name": "track_1m", "kind": "track", "n": 1_000_000, "hits": False},
        # Field and potential at every charge of the headline GEM workload: 1e6 charges, 60k cells.
        {"name": "field_gem_1m", "kind": "field", "mesh": "gem", "cells": 60_000, "n": 1_000_000, "groups": True},
        # Field on a probe set and the gradient of a loss on it (points, charges, cell densities).
        {"name": "probe_gradient", "kind": "probe", "cells": 30_000, "nt": 4096, "n": 100_000},
        # Electrode design: loss on the double GEM's axis, gradient with respect to the six voltages
        # (through the solve and its adjoint) and the charges.
        {"name": "voltage_gradient", "kind": "voltages", "cells": 11_000, "nt": 4096, "n": 20_000},
        # Set-up of a new geometry: assemble, factorise and solve the 60k-cell GEM.
        {"name": "bem_gem_60k", "kind": "bem", "mesh": "gem", "cells": 60_000, "precision": "bf16"},
        # The dynamic option: influence of the charges on the cells and the re-solve with the stored factors.
        {"name": "resolve_gem", "kind": "resolve", "mesh": "gem", "cells": 60_000, "n": 250_000},
        # Parameter sweep: 64 uneven chambers, one step of all of them as a captured graph.
        {"name": "batch_sweep", "kind": "batch", "chambers": 64, "n_max": 30_000},
        # Approximate N-body field of a large avalanche.
        {"name": "nbody_nn", "kind": "nn", "n": 300_000, "grid": 16},
        # Static field map of a plate chamber, built and interpolated at the charges.
        {"name": "field_map", "kind": "map", "cells": 2048, "nx": 100, "ny": 90, "nz": 80, "points": 500_000},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["steps", "steps", "track", "field", "probe", "voltages", "bem", "resolve", "batch", "nn", "map"])
    if kind == "steps":
        mesh = rng.choice(["plates", "plates", "gem"])
        return {"kind": kind, "mesh": mesh, "cells": _log(rng, 800, 40_000) if mesh == "gem" else _log(rng, 512, 8192),
                "n": _log(rng, 100, 60_000), "gas": rng.choice(["maxwell", "argon"]), "steps": rng.randint(1, 4),
                "groups": mesh == "gem" and rng.random() < 0.7}
    if kind == "track":
        return {"kind": kind, "n": _log(rng, 500, 1_000_000), "hits": rng.random() < 0.4}
    if kind == "field":
        mesh = rng.choice(["none", "plates", "gem"])
        return {"kind": kind, "mesh": mesh, "cells": _log(rng, 800, 40_000) if mesh == "gem" else _log(rng, 512, 8192),
                "n": _log(rng, 50, 300_000), "groups": mesh == "gem" and rng.random() < 0.7}
    if kind == "probe":
        return {"kind": kind, "cells": _log(rng, 800, 30_000), "nt": _log(rng, 64, 8192), "n": _log(rng, 100, 200_000)}
    if kind == "voltages":
        return {"kind": kind, "cells": _log(rng, 1600, 11_000), "nt": _log(rng, 64, 4096), "n": _log(rng, 100, 20_000)}
    if kind == "bem":
        precision = rng.choice(["bf16", "bf16", "bf16", "tf32", "fp32"])
        return {"kind": kind, "mesh": rng.choice(["plates", "gem"]),
                "cells": _log(rng, 800, 30_000 if precision == "bf16" else 8000), "precision": precision}
    if kind == "resolve":
        return {"kind": kind, "mesh": "gem", "cells": _log(rng, 800, 30_000), "n": _log(rng, 500, 250_000)}
    if kind == "batch":
        return {"kind": kind, "chambers": _log(rng, 2, 64), "n_max": _log(rng, 500, 30_000)}
    if kind == "nn":
        return {"kind": kind, "n": _log(rng, 1000, 300_000), "grid": rng.choice([8, 12, 16, 21, 32])}
    return {"kind": kind, "cells": _log(rng, 512, 4096), "nx": rng.randint(20, 110), "ny": rng.randint(20, 110),
            "nz": rng.randint(20, 80), "points": _log(rng, 1000, 1_000_000)}


# ---------------------------------------------------------------- geometry and charges
@functools.lru_cache(maxsize=None)
def _plates(cells):
    """Parallel plates of about `cells` triangles, 1 cm x 1 cm, 1 mm apart."""
    n = max(2, int(round(math.sqrt(cells / 4.0))))
    return inputs.parallel_plates(1e-2, 1e-3, n, ny=max(2, int(round(cells / (4.0 * n)))))


@functools.lru_cache(maxsize=None)
def _gem(cells):
    """Single-GEM patch of about `cells` triangles: 19, 7 or 1 holes."""
    geo = inputs.GemGeometry(rings=2 if cells >= 16_000 else 1 if cells >= 6000 else 0)
    return inputs.gem_mesh_target(cells, geo), geo


@functools.lru_cache(maxsize=None)
def _double_gem(cells):
    geo = inputs.DoubleGemGeometry(foil=inputs.GemGeometry(rings=1 if cells >= 10_600 else 0))
    return inputs.double_gem_mesh_target(cells, geo), geo


@functools.lru_cache(maxsize=None)
def _argon():
    return inputs.argon_like_gas()


def _gas(case):
    return inputs.maxwell_gas(1e12, 0.0) if case["gas"] == "maxwell" else _argon()


def _voltages(mesh, rng):
    """The mesh's voltages, each off its nominal value by up to 2 %."""
    return mesh.group_voltage * rng.uniform(0.98, 1.02, mesh.n_groups)


def _gem_cloud(geo, n, rng, z=(0.0,)):
    """n points in Gaussian clouds (20 um) on the hole axes, outside the foils centred at the heights z."""
    g = torch.Generator(DEV).manual_seed(int(rng.integers(1 << 62)))
    cen = torch.tensor(geo.hole_centres(), **F64)
    zt = torch.tensor(z, **F64)
    zk, zc = geo.t_kapton / 2, geo.t_kapton / 2 + geo.t_copper
    parts, have = [], 0
    while have < n:
        m = int((n - have) * 1.4) + 64
        h = torch.randint(len(cen), (m,), generator=g, device=DEV)
        f = torch.randint(len(zt), (m,), generator=g, device=DEV)
        p = torch.randn(m, 3, generator=g, **F64) * 20e-6
        p[:, :2] += cen[h]
        r = torch.cdist(p[:, :2], cen).amin(1)
        az = p[:, 2].abs()
        wall = torch.where(az < zk, geo.d_inner / 2 + (geo.d_outer - geo.d_inner) / 2 * az / zk, geo.d_outer / 2)
        p[:, 2] += zt[f]
        p = p[(az >= zc) | (r < wall)]
        parts.append(p)
        have += len(p)
    return torch.cat(parts)[:n].cpu().numpy()


def _charges(case, mesh, geo, rng):
    """Half electrons (Maxwellian), half cations; electrons only in the Maxwell-model gas."""
    n = case["n"]
    if case["mesh"] == "gem":
        pos = _gem_cloud(geo, n, rng)
        sp = (rng.random(n) < 0.5).astype(np.uint8)
    elif case.get("gas") == "maxwell":
        pos = inputs.uniform_box(rng, n, (0, 0, 2e-5), (1e-2, 1e-2, 9.8e-4))
        sp = np.zeros(n, np.uint8)
    else:
        ch = inputs.avalanche_snapshot(rng, n, gap=1e-3)
        ch.pos_q[:, 2] = np.clip(ch.pos_q[:, 2], 2e-5, 9.8e-4)
        return ch
    if case.get("gas") == "maxwell":
        sp[:] = 0
    vel = np.where((sp == 0)[:, None], inputs.maxwellian(rng, n, 1.0, inputs.M_ELECTRON), 0.0)
    return inputs.make_charges(pos, vel, sp)


def _mesh(case):
    return (_plates(case["cells"]), None) if case["mesh"] == "plates" else _gem(case["cells"])


class Context:
    """An obem context that goes with its owner."""

    def __init__(self, **kw):
        self.h = obem.obem_create(**kw)

    def __del__(self):
        if self.h is not None:
            obem.obem_destroy(self.h)
            self.h = None


def _solved(mesh, voltages, **kw):
    """A context holding the mesh, its BF16 factors and the solution, and the solution."""
    ctx = Context(**kw)
    obem.obem_mesh_load(ctx.h, mesh)
    obem.obem_bem_assemble(ctx.h, obem.OBEM_LU_BF16)
    sigma = torch.empty(mesh.n, dtype=torch.float32, device=DEV)
    obem.obem_bem_solve(ctx.h, voltages, sigma)
    return ctx, sigma


def _cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


class Snapshot:
    """A device state and the copy that every pass starts from."""

    def __init__(self, st):
        self.st = st
        self.names = [k for k, v in vars(st).items() if isinstance(v, torch.Tensor)]
        self.copy = {k: getattr(st, k).clone() for k in self.names}

    def restore(self):
        for k in self.names:
            getattr(self.st, k).copy_(self.copy[k])

    def outputs(self):
        return {k: getattr(self.st, k) for k in self.names}


def _stat_counts(stats, steps):
    """The whole numbers of obem_step_stats (12 int32, one int64) of `steps` records."""
    s = stats.view(steps, obem.STATS_BYTES)
    return {"counts": s.view(torch.int32)[:, :12], "trials": s.view(torch.int64)[:, 6:7]}


# ---------------------------------------------------------------- inputs
def prepare(case, seed):
    rng = np.random.default_rng([seed, 977])
    return globals()["_prepare_" + case["kind"]](case, rng)


def run(state):
    return state["run"](state)


def _prepare_steps(case, rng):
    mesh, geo = _mesh(case)
    ch = _charges(case, mesh, geo, rng)
    cap = int(case["n"] * 1.2) + 1024
    z = (geo.z_anode, geo.z_drift) if geo else (0.0, 1e-3)
    flags = obem.OBEM_STEP_SPACE_CHARGE | obem.OBEM_STEP_CELL_FIELD | (obem.OBEM_STEP_CELL_GROUPS if case["groups"] else 0)
    ctx, sigma = _solved(mesh, _voltages(mesh, rng) if geo else np.array([0.0, rng.uniform(50.0, 1000.0)]),
                         capacity=cap, dt=1e-12, seed=int(rng.integers(1 << 31)), softening=1e-9, z_lo=z[0], z_hi=z[1],
                         beta=-1.0 if case["gas"] == "maxwell" else 1e-13, flags=flags)
    obem.obem_gas_load(ctx.h, _gas(case))
    st = obem.DeviceState(cap, DEV)
    st.upload(ch)
    return {"run": _run_steps, "ctx": ctx, "snap": Snapshot(st), "steps": case["steps"],
            "stats": torch.zeros(case["steps"], obem.STATS_BYTES, dtype=torch.uint8, device=DEV)}


def _run_steps(s):
    s["snap"].restore()
    for k in range(s["steps"]):
        obem.obem_step(s["ctx"].h, s["snap"].st, k, s["stats"][k])
    return {**s["snap"].outputs(), **_stat_counts(s["stats"], s["steps"])}


def _prepare_track(case, rng):
    n = case["n"]
    cap = int(n * 1.2) + 1024
    flags = obem.OBEM_STEP_SURFACE_HITS if case["hits"] else 0
    if case["hits"]:
        mesh, geo = _gem(16_000)
        ch = _charges({"n": n, "mesh": "gem"}, mesh, geo, rng)
        z = (geo.z_anode, geo.z_drift)
    else:
        mesh, ch, z = None, inputs.avalanche_snapshot(rng, n), (0.0, 2e-3)
        ch.pos_q[:, 2] = np.clip(ch.pos_q[:, 2], 4e-5, 1.96e-3)
    el = ch.species == inputs.SP_ELECTRON
    ch.vel[el, :3] *= 2.0                       # kT 4 eV: an avalanche's electrons
    ctx = Context(capacity=cap, dt=1e-12, seed=int(rng.integers(1 << 31)), softening=1e-9, z_lo=z[0], z_hi=z[1],
                  beta=1e-13, flags=flags)
    obem.obem_gas_load(ctx.h, _argon())
    if mesh is not None:
        obem.obem_mesh_load(ctx.h, mesh)
    E = np.zeros((cap, 4), np.float32)
    E[:n, :3] = rng.normal(0.0, 1e5, (n, 3))
    E[:n, 2] += 1e6
    st = obem.DeviceState(cap, DEV)
    st.upload(ch)
    return {"run": _run_track, "ctx": ctx, "snap": Snapshot(st), "E": _cuda(E),
            "stats": torch.zeros(obem.STATS_BYTES, dtype=torch.uint8, device=DEV),
            "np": mesh.n if mesh is not None else 0}


def _run_track(s):
    s["snap"].restore()
    obem.obem_step(s["ctx"].h, s["snap"].st, 3, s["stats"], E_in=s["E"])
    out = {**s["snap"].outputs(), **_stat_counts(s["stats"], 1), "moments": s["stats"].view(torch.float64)[7:20]}
    if s["np"]:
        out["deposits"] = obem.obem_surface_charge(s["ctx"].h, s["np"], reset=True)
    return out


def _prepare_field(case, rng):
    n, sigma, mesh = case["n"], None, None
    flags = obem.OBEM_STEP_CELL_GROUPS if case["groups"] else 0
    if case["mesh"] != "none":
        mesh, geo = _mesh(case)
        # densities from a solve of their own; the evaluating context keeps the mesh only
        solver, sigma = _solved(mesh, _voltages(mesh, rng) if geo else np.array([0.0, rng.uniform(50.0, 1000.0)]),
                                capacity=16, dt=1e-12)
        del solver
        ch = _charges(case, mesh, geo, rng)
    else:
        ch = inputs.avalanche_snapshot(rng, n)
    ctx = Context(capacity=n, dt=1e-12, flags=flags)
    if mesh is not None:
        obem.obem_mesh_load(ctx.h, mesh)
    return {"run": _run_field, "ctx": ctx, "q": _cuda(ch.pos_q), "sigma": sigma,
            "E": torch.zeros(n, 4, dtype=torch.float32, device=DEV)}


def _run_field(s):
    obem.obem_field_eval(s["ctx"].h, s["q"], s["E"], sources=s["q"], self_exclude=True, sigma=s["sigma"])
    return {"E": s["E"]}


def _probe_points(geo, nt, rng):
    """Points on and around the central hole's axis, between the planes."""
    z = np.sort(rng.uniform(geo.z_anode, geo.z_drift, nt))
    return np.column_stack([rng.normal(0.0, 4e-6, nt), rng.normal(0.0, 4e-6, nt), z, np.zeros(nt)]).astype(np.float32)


def _prepare_probe(case, rng):
    mesh, geo = _gem(case["cells"])
    solver, sigma = _solved(mesh, _voltages(mesh, rng), capacity=16, dt=1e-12)
    del solver
    ch = _charges({"n": case["n"], "mesh": "gem"}, mesh, geo, rng)
    ctx = Context(capacity=max(case["n"], case["nt"]), dt=1e-12)
    obem.obem_mesh_load(ctx.h, mesh)
    leaf = lambda t: t.requires_grad_(True)  # noqa: E731
    return {"run": _run_probe, "ctx": ctx, "x": leaf(_cuda(_probe_points(geo, case["nt"], rng))),
            "q": leaf(_cuda(ch.pos_q)), "sigma": leaf(sigma)}


def _run_probe(s):
    E = obem.field_eval(s["ctx"].h, s["x"], s["q"], s["sigma"])
    loss = (E[:, :3] ** 2).mean() * 1e-8
    dx, dq, ds = torch.autograd.grad(loss, (s["x"], s["q"], s["sigma"]))
    return {"E": E.detach(), "dx": dx, "dq_pos": dq[:, :3], "dq_charge": dq[:, 3], "dsigma": ds}


def _prepare_voltages(case, rng):
    mesh, geo = _double_gem(case["cells"])
    V = torch.tensor(_voltages(mesh, rng), dtype=torch.float32)
    ctx, _ = _solved(mesh, V.double().numpy(), capacity=max(case["n"], case["nt"]), dt=1e-12)
    f = geo.foil
    pos = _gem_cloud(f, case["n"], rng, (geo.z_upper, geo.z_lower))
    ch = inputs.make_charges(pos, np.zeros_like(pos), (rng.random(case["n"]) < 0.5).astype(np.uint8))
    return {"run": _run_voltages, "ctx": ctx, "V": V.requires_grad_(True), "np": mesh.n,
            "x": _cuda(_probe_points(geo, case["nt"], rng)), "q": _cuda(ch.pos_q).requires_grad_(True)}


def _run_voltages(s):
    sigma = obem.bem_solve(s["ctx"].h, s["V"], s["np"])
    E = obem.field_eval(s["ctx"].h, s["x"], s["q"], sigma)
    loss = (E[:, :3] ** 2).mean() * 1e-8
    dV, dq = torch.autograd.grad(loss, (s["V"], s["q"]))
    return {"sigma": sigma.detach(), "E": E.detach(), "dV": dV, "dq_pos": dq[:, :3], "dq_charge": dq[:, 3]}


def _prepare_bem(case, rng):
    mesh, geo = _mesh(case)
    ctx = Context(capacity=16, dt=1e-12)
    obem.obem_mesh_load(ctx.h, mesh)
    V = _voltages(mesh, rng) if geo else np.array([0.0, rng.uniform(50.0, 1000.0)])
    return {"run": _run_bem, "ctx": ctx, "V": V, "precision": PRECISION[case["precision"]],
            "sigma": torch.zeros(mesh.n, dtype=torch.float32, device=DEV)}


def _run_bem(s):
    obem.obem_bem_assemble(s["ctx"].h, s["precision"])
    obem.obem_bem_solve(s["ctx"].h, s["V"], s["sigma"])
    return {"sigma": s["sigma"]}


def _prepare_resolve(case, rng):
    mesh, geo = _mesh(case)
    V = _voltages(mesh, rng)
    ctx, sigma = _solved(mesh, V, capacity=16, dt=1e-12)
    ch = _charges(case, mesh, geo, rng)
    # each charge stands for 1000 (a dense avalanche's space charge)
    ch.pos_q[:, 3] *= np.float32(1000.0)
    return {"run": _run_resolve, "ctx": ctx, "V": V, "q": _cuda(ch.pos_q), "sigma": sigma,
            "drhs": torch.zeros(mesh.n, dtype=torch.float32, device=DEV)}


def _run_resolve(s):
    obem.obem_influence_rhs(s["ctx"].h, s["q"], s["drhs"])
    obem.obem_bem_solve(s["ctx"].h, s["V"], s["sigma"], drhs=s["drhs"])
    return {"drhs": s["drhs"], "sigma": s["sigma"]}


def _prepare_batch(case, rng):
    flags = obem.OBEM_STEP_SPACE_CHARGE | obem.OBEM_STEP_CELL_FIELD
    ctx = Context(capacity=16, dt=1e-12, softening=1e-7, beta=1e-13, flags=flags)
    obem.obem_gas_load(ctx.h, _argon())
    sets, gaps, cells = [], [], []
    for k in range(case["chambers"]):
        gap = rng.uniform(0.5e-3, 3e-3)
        # charges log-uniform in 1e2 .. n_max, small and large chambers mixed
        u = ((k * 29) % case["chambers"] + 0.5) / case["chambers"]
        ch = inputs.avalanche_snapshot(rng, int(round(100.0 * (case["n_max"] / 100.0) ** u)), gap=gap)
        ch.pos_q[:, 2] = np.clip(ch.pos_q[:, 2], 0.02 * gap, 0.98 * gap)
        tri = _plates((1024, 1600, 2304, 4096)[k % 4]).tri.copy()
        top = tri[:, 0, 2] > 0
        tri[top, :, 2] = gap
        # the plates' own density: E = V / gap, the sheet carrying both faces
        e = 10.0 ** rng.uniform(4.0, 6.5)
        sigma = np.where(top, EPS0 * e, -EPS0 * e).astype(np.float32)
        sets.append(ch)
        gaps.append(gap)
        cells.append((tri, sigma))
    caps = [max(int(1.5 * c.n), 256) for c in sets]
    b = obem.Batch(ctx.h, caps, [0.0] * len(caps), gaps, rng.integers(1, 1 << 31, len(caps)))
    for k, (tri, sigma) in enumerate(cells):
        b.cells(k, tri, sigma)
    st = b.state(DEV)
    st.upload(sets)
    return {"run": _run_batch, "batch": _Batch(b, ctx), "snap": Snapshot(st), "nb": len(caps),
            "step": torch.zeros(1, dtype=torch.int32, device=DEV), "stats": obem.new_batch_stats(len(caps), DEV)}


class _Batch:
    def __init__(self, b, ctx):
        self.b, self.ctx = b, ctx

    def __del__(self):
        self.b.destroy()


def _run_batch(s):
    s["snap"].restore()
    s["step"].zero_()
    s["batch"].b.step_graph(s["snap"].st, s["step"], s["stats"])
    return {**s["snap"].outputs(), "step": s["step"], **_stat_counts(s["stats"], s["nb"])}


def _prepare_nn(case, rng):
    ch = inputs.avalanche_snapshot(rng, case["n"])
    return {"run": _run_nn, "ctx": Context(capacity=case["n"], dt=1e-12), "q": _cuda(ch.pos_q), "grid": case["grid"],
            "E": torch.zeros(case["n"], 4, dtype=torch.float32, device=DEV)}


def _run_nn(s):
    obem.obem_nbody_nn_eval(s["ctx"].h, s["q"], s["E"], s["grid"], softening=1e-9)
    return {"E": s["E"]}


MAP_BOX = (np.array([2e-3, 2.2e-3, 1.5e-4]), np.array([7.7e-3, 8e-3, 8.6e-4]))


def _prepare_map(case, rng):
    mesh = _plates(case["cells"])
    ctx, sigma = _solved(mesh, np.array([0.0, rng.uniform(50.0, 1000.0)]), capacity=16, dt=1e-12)
    pts = np.zeros((case["points"], 4), np.float32)
    pts[:, :3] = rng.uniform(MAP_BOX[0], MAP_BOX[1], (case["points"], 3))
    return {"run": _run_map, "ctx": ctx, "sigma": sigma, "pts": _cuda(pts), "dims": (case["nx"], case["ny"], case["nz"]),
            "E": torch.zeros(case["points"], 4, dtype=torch.float32, device=DEV)}


def _run_map(s):
    obem.obem_fieldmap_build(s["ctx"].h, MAP_BOX[0], MAP_BOX[1], s["dims"], s["sigma"])
    obem.obem_fieldmap_eval(s["ctx"].h, s["pts"], s["E"])
    return {"E": s["E"]}


# ---------------------------------------------------------------- necessary work
def work(case):
    """Bytes: inputs read once, outputs written once.  Flops: 18 per evaluated
    charge pair (an unordered pair once where both its charges are targets) and
    per cell seen from a point (one quadrature point), 2/3 n^3 for a
    factorisation, 2 n^2 per solve."""
    k, n = case["kind"], case.get("n", 0)
    m = {"mesh": "none", **case}
    c = 0 if k in ("track", "nn", "batch") or (k == "field" and m["mesh"] == "none") else case["cells"]
    cell, charge = 84.0, 41.0
    if k == "steps":
        return {"bytes": case["steps"] * (2 * charge * n + cell * c), "flops": case["steps"] * 18.0 * (n * n / 2.0 + n * c)}
    if k == "track":
        return {"bytes": (2 * charge + 16) * n, "flops": 500.0 * n}
    if k == "field":
        return {"bytes": 32.0 * n + cell * c, "flops": 18.0 * (n * n / 2.0 + n * c)}
    if k in ("probe", "voltages"):
        nt = case["nt"]
        solve = 2 * (4.0 * c * c) if k == "voltages" else 0.0
        return {"bytes": 48.0 * nt + 32.0 * n + 2 * cell * c + solve, "flops": 2 * 18.0 * nt * (n + c) + solve}
    if k == "bem":
        return {"bytes": cell * c + 4.0 * c, "flops": 2.0 / 3.0 * c ** 3 + 18.0 * c * c}
    if k == "resolve":
        return {"bytes": 16.0 * n + cell * c + 4.0 * c * c, "flops": 18.0 * n * c + 2.0 * c * c}
    if k == "batch":
        mean = (case["n_max"] - 100.0) / math.log(case["n_max"] / 100.0)
        mean2 = (case["n_max"] ** 2 - 1e4) / (2.0 * math.log(case["n_max"] / 100.0))
        return {"bytes": case["chambers"] * (2 * charge * mean + cell * 2256),
                "flops": case["chambers"] * 18.0 * (mean2 / 2.0 + 2256 * mean)}
    if k == "nn":
        return {"bytes": 32.0 * n, "flops": 18.0 * n * 2.0 * case["grid"] ** 3}
    nodes = case["nx"] * case["ny"] * case["nz"]
    return {"bytes": 32.0 * case["points"] + 16.0 * nodes + cell * c, "flops": 18.0 * nodes * c + 64.0 * case["points"]}


# ---------------------------------------------------------------- the same in 64 bits
def _tri_integrals(tri, x):
    """Potential and field of a unit density on flat triangles tri [m, 3, 3] at
    points x [p, 1, 3]: phi [p, m], F [p, m, 3].  Edge logarithms and the solid
    angle; the principal value in a triangle's plane."""
    dot = lambda a, b: (a * b).sum(-1)  # noqa: E731
    nrm = torch.linalg.cross(tri[:, 1] - tri[:, 0], tri[:, 2] - tri[:, 0])
    a2 = nrm.norm(dim=-1)
    nrm = nrm / a2[:, None]
    a = [tri[None, :, i] - x for i in range(3)]
    R = [v.norm(dim=-1) for v in a]
    h = -dot(a[0], nrm)
    phi, F = 0.0, 0.0
    for i in range(3):
        j = (i + 1) % 3
        t = tri[:, j] - tri[:, i]
        t = t / t.norm(dim=-1, keepdim=True)
        u = torch.linalg.cross(t, nrm)
        lm, lp, p0 = dot(a[i], t), dot(a[j], t), dot(a[i], u)
        num = torch.where(lm >= 0, R[j] + lp, torch.where(lp <= 0, R[i] - lm, (R[j] + lp) * (R[i] - lm)))
        den = torch.where(lm >= 0, R[i] + lm, torch.where(lp <= 0, R[j] - lp, p0 * p0 + h * h))
        L = torch.log(num / den)
        phi = phi + p0 * L
        F = F + u * L[..., None]
    D = R[0] * R[1] * R[2] + dot(a[0], a[1]) * R[2] + dot(a[0], a[2]) * R[1] + dot(a[1], a[2]) * R[0]
    om = torch.where(h == 0, torch.zeros_like(h), 2.0 * torch.atan2(a2 * h, D))
    return phi - h * om, F + nrm * om[..., None]


def _cell_field(tri, sigma, x, pairs=4_000_000):
    """(Ex, Ey, Ez, V) at points x [n, 3] of the cells."""
    out = torch.zeros(len(x), 4, **F64)
    step = max(1, pairs // len(tri))
    for k in range(0, len(x), step):
        phi, F = _tri_integrals(tri, x[k:k + step, None])
        out[k:k + step, :3] = KC * torch.einsum("pmc,m->pc", F, sigma)
        out[k:k + step, 3] = KC * (phi @ sigma)
    return out


def _charge_field(q, x, skip_self, pairs=32_000_000):
    """(Ex, Ey, Ez, V) at points x [n, 3] of the charges q [m, 4]."""
    out = torch.zeros(len(x), 4, **F64)
    step = max(1, pairs // len(q))
    for k in range(0, len(x), step):
        d = [x[k:k + step, c, None] - q[None, :, c] for c in range(3)]
        r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2]
        if skip_self:
            r2[torch.arange(len(r2)), torch.arange(k, k + len(r2))] = math.inf
        w = KC * q[:, 3] * r2.rsqrt()
        out[k:k + step, 3] = w.sum(1)
        w = w / r2
        for c in range(3):
            out[k:k + step, c] = (w * d[c]).sum(1)
    return out


def _matrix(mesh, pairs=4_000_000):
    """The collocation matrix: potential rows on electrode cells, normal-field rows on dielectric cells."""
    tri = torch.tensor(mesh.tri, **F64)
    n = len(tri)
    cen = tri.mean(1)
    nrm = torch.linalg.cross(tri[:, 1] - tri[:, 0], tri[:, 2] - tri[:, 0])
    nrm = nrm / nrm.norm(dim=-1, keepdim=True)
    em, ep = torch.tensor(mesh.eps_minus, **F64), torch.tensor(mesh.eps_plus, **F64)
    electrode = torch.tensor(mesh.kind == inputs.KIND_ELECTRODE, device=DEV)
    A = torch.empty(n, n, **F64)
    step = max(1, pairs // n)
    for k in range(0, n, step):
        phi, F = _tri_integrals(tri, cen[k:k + step, None])
        rows = torch.arange(k, k + len(phi), device=DEV)
        W = (ep - em)[rows, None] / (4.0 * math.pi) * torch.einsum("pmc,pc->pm", F, nrm[rows])
        W[rows - k, rows] = (0.5 * (ep + em))[rows]
        A[rows] = torch.where(electrode[rows, None], KC * phi, W)
    return A


def _rhs(mesh, V):
    b = torch.zeros(mesh.n, **F64)
    group = torch.tensor(mesh.group, device=DEV).long().clamp(min=0)
    electrode = torch.tensor(mesh.kind == inputs.KIND_ELECTRODE, device=DEV)
    return torch.where(electrode, torch.as_tensor(V, **F64)[group], b)


def _influence(mesh, q, pairs=4_000_000):
    """Right-hand-side correction: minus the charges' mean potential on electrode
    cells, minus (eps+ - eps-) eps0 times their mean normal field on dielectric cells."""
    tri = torch.tensor(mesh.tri, **F64)
    S = torch.zeros(mesh.n, 4, **F64)
    step = max(1, pairs // mesh.n)
    for k in range(0, len(q), step):
        phi, F = _tri_integrals(tri, q[k:k + step, None, :3])
        S[:, 0] += KC * (q[k:k + step, 3] @ phi)
        S[:, 1:] += KC * torch.einsum("pmc,p->mc", F, q[k:k + step, 3])
    nrm = torch.linalg.cross(tri[:, 1] - tri[:, 0], tri[:, 2] - tri[:, 0])
    area = 0.5 * nrm.norm(dim=-1)
    nrm = nrm / (2.0 * area[:, None])
    eps = torch.tensor(mesh.eps_plus - mesh.eps_minus, **F64)
    electrode = torch.tensor(mesh.kind == inputs.KIND_ELECTRODE, device=DEV)
    return torch.where(electrode, -S[:, 0], eps * EPS0 * (S[:, 1:] * nrm).sum(-1)) / area


def _probe_grads(x, q, tri, sigma, E, want_x=True, pairs=1_000_000):
    """Gradients of 1e-8 mean |E|^2 with respect to the points (x, y, z, 0), the
    charges (x, y, z, q) and the cell densities."""
    g = E[:, :3] * (2e-8 / (3 * len(x)))
    dx = torch.zeros(len(x), 4, **F64)
    dq = torch.zeros(len(q), 4, **F64)
    ds = torch.zeros(len(tri), **F64)
    step = max(1, 8_000_000 // len(q))
    for k in range(0, len(x), step):
        gk = g[k:k + step, None]
        d = x[k:k + step, None] - q[None, :, :3]
        r2 = (d * d).sum(-1)
        dg = (d * gk).sum(-1)
        i3 = KC * r2 ** -1.5
        T = i3[..., None] * (gk - (3.0 * dg / r2)[..., None] * d)
        dq[:, :3] -= (T * q[None, :, 3:]).sum(0)
        dq[:, 3] += (i3 * dg).sum(0)
        dx[k:k + step, :3] += (T * q[None, :, 3:]).sum(1)
    step = max(1, pairs // len(tri))
    for k in range(0, len(x), step):
        xk = x[k:k + step].clone().requires_grad_(want_x)
        with torch.enable_grad():
            _, F = _tri_integrals(tri, xk[:, None])
            w = KC * (F * g[k:k + step, None]).sum(-1)
            if want_x:
                dx[k:k + step, :3] += torch.autograd.grad(w @ sigma, xk, torch.ones(len(xk), **F64))[0]
        ds += w.detach().sum(0)
    return dx, dq, ds


def exact(case, seed):
    f = globals().get("_exact_" + case["kind"])
    if f is None or not torch.cuda.is_available():
        return None
    with torch.no_grad():
        return f(case, seed)


def _exact_field(case, seed):
    if 1.0 * case["n"] ** 2 + (20.0 * case["n"] * case["cells"] if case["mesh"] != "none" else 0.0) > EXACT_PAIRS:
        return None
    s = prepare(case, seed)
    q = s["q"].double()
    E = _charge_field(q, q[:, :3], True)
    if s["sigma"] is not None:
        E += _cell_field(torch.tensor(_mesh(case)[0].tri, **F64), s["sigma"].double(), q[:, :3])
    return {"E": E}


def _exact_probe(case, seed):
    s = prepare(case, seed)
    tri = torch.tensor(_gem(case["cells"])[0].tri, **F64)
    x, q, sigma = s["x"].detach().double()[:, :3], s["q"].detach().double(), s["sigma"].detach().double()
    E = _charge_field(q, x, False) + _cell_field(tri, sigma, x)
    dx, dq, ds = _probe_grads(x, q, tri, sigma, E)
    return {"E": E, "dx": dx, "dq_pos": dq[:, :3], "dq_charge": dq[:, 3], "dsigma": ds}


def _exact_voltages(case, seed):
    s = prepare(case, seed)
    mesh = _double_gem(case["cells"])[0]
    tri = torch.tensor(mesh.tri, **F64)
    x, q = s["x"].double()[:, :3], s["q"].detach().double()
    LU = torch.linalg.lu_factor(_matrix(mesh))
    sigma = torch.linalg.lu_solve(*LU, _rhs(mesh, s["V"].detach().double().to(DEV))[:, None])[:, 0]
    E = _charge_field(q, x, False) + _cell_field(tri, sigma, x)
    _, dq, ds = _probe_grads(x, q, tri, sigma, E, want_x=False)
    mu = torch.linalg.lu_solve(*LU, ds[:, None], adjoint=True)[:, 0]
    electrode = torch.tensor(mesh.kind == inputs.KIND_ELECTRODE, device=DEV)
    group = torch.tensor(mesh.group, device=DEV).long()
    dV = torch.zeros(mesh.n_groups, **F64).index_add_(0, group[electrode], mu[electrode])
    return {"sigma": sigma, "E": E, "dV": dV, "dq_pos": dq[:, :3], "dq_charge": dq[:, 3]}


def _exact_bem(case, seed):
    mesh = _mesh(case)[0]
    if mesh.n > EXACT_CELLS:
        return None
    V = prepare(case, seed)["V"]
    return {"sigma": torch.linalg.solve(_matrix(mesh), _rhs(mesh, V))}


def _exact_resolve(case, seed):
    mesh = _mesh(case)[0]
    if 1.0 * mesh.n * case["n"] > 8e9:
        return None
    s = prepare(case, seed)
    drhs = _influence(mesh, s["q"].double())
    if mesh.n > EXACT_CELLS:
        return {"drhs": drhs, "sigma": None}
    return {"drhs": drhs, "sigma": torch.linalg.solve(_matrix(mesh), _rhs(mesh, s["V"]) + drhs)}


def _exact_map(case, seed):
    if 1.0 * case["nx"] * case["ny"] * case["nz"] * case["cells"] > 8e9:
        return None
    s = prepare(case, seed)
    dims = [case["nx"], case["ny"], case["nz"]]
    lo, hi = torch.tensor(MAP_BOX[0], **F64), torch.tensor(MAP_BOX[1], **F64)
    step = (hi - lo) / (torch.tensor(dims, **F64) - 1)
    axes = [lo[a] + torch.arange(dims[a], **F64) * step[a] for a in range(3)]
    nodes = torch.stack(torch.meshgrid(*axes, indexing="ij"), -1).reshape(-1, 3)
    N = _cell_field(torch.tensor(_plates(case["cells"]).tri, **F64), s["sigma"].double(), nodes).reshape(*dims, 4)
    f = (s["pts"].double()[:, :3] - lo) / step
    top = torch.tensor(dims, device=DEV) - 2
    i = torch.minimum(f.floor().long().clamp(min=0), top)
    t = (f - i).clamp(0.0, 1.0)
    E = torch.zeros(len(t), 4, **F64)
    for c in range(8):
        o = [(c >> a) & 1 for a in range(3)]
        w = math.prod([t[:, a] if o[a] else 1.0 - t[:, a] for a in range(3)])
        E += w[:, None] * N[i[:, 0] + o[0], i[:, 1] + o[1], i[:, 2] + o[2]]
    return {"E": E}


def _exact_nn(case, seed):
    """Exact softened sums over the 27 cells around a charge, the other cells'
    positive and negative charge at their charge-weighted centres."""
    s = prepare(case, seed)
    q32, G, eps2 = s["q"], case["grid"], 1e-18
    p = q32[:, :3]
    lo = p.amin(0)
    inv = torch.tensor(np.float32(G) / np.float32((p.amax(0) - lo).amax().item()), device=DEV)
    cell = ((p - lo) * inv).floor().long().clamp(0, G - 1)
    flat = (cell[:, 2] * G + cell[:, 1]) * G + cell[:, 0]
    order = torch.argsort(flat, stable=True)
    q, flat = q32.double()[order], flat[order]
    nc = G ** 3
    start = torch.searchsorted(flat, torch.arange(nc + 1, device=DEV)).tolist()
    centre = []
    for part in (q[:, 3].clamp(min=0.0), q[:, 3].clamp(max=0.0)):
        Q = torch.zeros(nc, **F64).index_add_(0, flat, part)
        C = torch.zeros(nc, 3, **F64).index_add_(0, flat, part[:, None] * q[:, :3])
        centre.append(torch.cat([C / torch.where(Q == 0, 1.0, Q)[:, None], Q[:, None]], 1))
    centre = torch.stack(centre)                                    # [2, nc, 4]

    def add(out, x, src, own=None):
        d = [x[:, c, None] - src[None, :, c] for c in range(3)]
        r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2] + eps2
        w = KC * src[:, 3] * r2 ** -1.5
        if own is not None:
            w[torch.arange(len(x)), own] = 0.0
        for c in range(3):
            out[:, c] += (w * d[c]).sum(1)

    E = torch.zeros(len(q), 4, **F64)
    every = torch.arange(nc, device=DEV)
    xyz = torch.stack([every % G, every // G % G, every // (G * G)], 1)
    for c in range(nc):
        a, b = start[c], start[c + 1]
        if a == b:
            continue
        cx, cy, cz = c % G, c // G % G, c // (G * G)
        near, own = [], None
        for z in range(max(0, cz - 1), min(G, cz + 2)):
            for y in range(max(0, cy - 1), min(G, cy + 2)):
                r = (z * G + y) * G
                k0, k1 = start[r + max(0, cx - 1)], start[r + min(G, cx + 2)]
                if (y, z) == (cy, cz):
                    own = sum(map(len, near)) + a - k0
                near.append(q[k0:k1])
        near = torch.cat(near)
        far = centre[:, ((xyz - xyz[c]).abs() > 1).any(1)].reshape(-1, 4)
        far = far[far[:, 3] != 0]
        step = max(1, 16_000_000 // (len(near) + len(far)))
        for k in range(a, b, step):
            m = min(b, k + step)
            add(E[k:m], q[k:m], near, own + torch.arange(k - a, m - a, device=DEV))
            add(E[k:m], q[k:m], far)
    out = torch.empty_like(E)
    out[order] = E
    return {"E": out}
