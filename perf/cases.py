"""Performance cases of the coupled D3Q19 lattice Boltzmann / rigid-body step.

Each case is one call (or one short series of calls) that a user's program
makes over and over through the public entry points: ``Lattice.step`` with a
read of the body states and of a field, ``Ensemble.step`` over many boxes,
``swimmer_run`` with its backward pass, and the allocation-free momentum
exchange of the C ABI.  Sizes come from this repository's workloads
(``workloads.py``, ``design_study.py``), or are generic boxes between them.

``exact`` restates the method in plain torch in 64 bits (gathers and rolls, no
kernel of this repository) and differentiates it with torch's own autograd.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

from paper_1108_0786_gb300 import autograd, design_study, lbm, workloads as wl

# ---- the cases ---------------------------------------------------------------


def listed():
    return [
        # a caller that owns its device memory asks for force and torque of the
        # three spheres of one small swimmer: the smallest call, two short kernels
        {"name": "static_force_48", "kind": "static", "nx": 48, "ny": 48, "nz": 48, "bodies": 3, "radius": 4.0,
         "half_width": 6, "bc": 7},
        # a controller or live view: one coupled step, then the body states and
        # the velocity field (one ensemble-sized box, a swimmer of radius 3)
        {"name": "control_step_48_f32", "kind": "step", "flow": "box", "nx": 48, "ny": 48, "nz": 48, "radius": 3.0,
         "capsules": False, "precision": "f32", "warm": 32, "steps": 1, "field": "u", "tuned": False},
        # the 32^3 FP64 swimmer of the parity configuration, 64 steps a read
        {"name": "swimmer_32_f64", "kind": "step", "flow": "box", "nx": 32, "ny": 32, "nz": 32, "radius": 3.0,
         "capsules": False, "precision": "f64", "warm": 32, "steps": 64, "field": "pop", "tuned": False},
        # the channel swimmer (128 x 64 x 64, walls, body force), FP32 and FP16
        {"name": "channel_f32", "kind": "step", "flow": "channel", "nx": 128, "ny": 64, "nz": 64, "radius": 6.0,
         "capsules": False, "precision": "f32", "warm": 32, "steps": 64, "field": "pop", "tuned": False},
        {"name": "channel_f16", "kind": "step", "flow": "channel", "nx": 128, "ny": 64, "nz": 64, "radius": 6.0,
         "capsules": False, "precision": "f16", "warm": 32, "steps": 64, "field": "pop", "tuned": False},
        # one point of the design study: 100 x 100 x 200 channel, perpendicular
        # capsules, averaged loads, the density and velocity written out
        {"name": "study_f32", "kind": "step", "flow": "study", "nx": 100, "ny": 100, "nz": 200, "radius": 4.0,
         "capsules": True, "precision": "f32", "warm": 64, "steps": 32, "field": "rho_u", "tuned": False},
        # an odd, ragged box of several swimmers in FP64 (no shape tuning)
        {"name": "ragged_swarm_f64", "kind": "step", "flow": "swarm", "nx": 203, "ny": 149, "nz": 131, "radius": 4.0,
         "capsules": True, "precision": "f64", "warm": 16, "steps": 8, "field": "pop", "tuned": False},
        # the throughput workload: 512 x 256 x 256, 8 swimmers, in the three
        # storage types used at that size
        {"name": "swarm_f32", "kind": "step", "flow": "swarm", "nx": 512, "ny": 256, "nz": 256, "radius": 4.0,
         "capsules": True, "precision": "f32", "warm": 32, "steps": 16, "field": "pop", "tuned": True},
        {"name": "swarm_f16", "kind": "step", "flow": "swarm", "nx": 512, "ny": 256, "nz": 256, "radius": 4.0,
         "capsules": True, "precision": "f16", "warm": 32, "steps": 16, "field": "pop", "tuned": True},
        {"name": "swarm_bf16", "kind": "step", "flow": "swarm", "nx": 512, "ny": 256, "nz": 256, "radius": 4.0,
         "capsules": True, "precision": "bf16", "warm": 32, "steps": 16, "field": "pop", "tuned": True},
        # half of the 96-box ensemble, one chunk of steps
        {"name": "ensemble_48_f32", "kind": "ensemble", "members": 48, "edge_max": 96, "precision": "f32", "warm": 16,
         "steps": 32},
        # one training step of the gradient study (96 x 48 x 48), forward and backward
        {"name": "gradient_f32", "kind": "gradient", "nx": 96, "ny": 48, "nz": 48, "capsules": False,
         "precision": "f32", "steps": 256, "segment": 64},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("static", "box", "box", "channel", "study", "swarm", "swarm", "ensemble", "gradient"))
    prec = rng.choice(("f64", "f32", "f32", "f16", "bf16"))
    if kind == "static":
        radius = rng.uniform(3.0, 12.0)
        n = [_log_int(rng, 4 * math.ceil(radius) + 12, 160) for _ in range(3)]
        room = math.prod(v // (2 * math.ceil(radius) + 4) for v in n)
        return {"kind": "static", "nx": n[0], "ny": n[1], "nz": n[2], "bodies": min(room, rng.randint(1, 24)),
                "radius": radius, "half_width": math.ceil(radius) + 2, "bc": rng.choice((7, 7, 4, 1))}
    if kind == "ensemble":
        return {"kind": "ensemble", "members": _log_int(rng, 2, 12 if prec == "f64" else 48),
                "edge_max": rng.choice((48, 64, 80, 96)), "precision": prec, "warm": 16,
                "steps": rng.choice((16, 32, 33, 47))}
    if kind == "gradient":
        # spheres: the capsule variant's rotational mode amplifies round-off
        return {"kind": "gradient", "nx": rng.randint(56, 96), "ny": rng.randint(32, 48), "nz": rng.randint(32, 48),
                "capsules": False, "precision": rng.choice(("f64", "f32")), "steps": rng.randint(64, 256),
                "segment": rng.choice((16, 32, 64))}
    steps = _log_int(rng, 1, 64)
    out = {"kind": "step", "precision": prec, "warm": rng.randint(8, 40), "tuned": rng.random() < 0.3,
           "field": rng.choice(("pop", "pop", "u", "rho_u")) if prec == "f32" else "pop"}
    if kind == "box":
        radius = rng.choice((3.0, 4.0, 6.0))
        capsules = rng.random() < 0.5
        half = radius * (2 if capsules else 1)
        side = 2 * (math.ceil(half) + 4) + 1
        out |= {"flow": "box", "nx": _log_int(rng, max(side, math.ceil(6 * half) + 14), 256),
                "ny": _log_int(rng, side, 192), "nz": _log_int(rng, side, 192), "radius": radius, "capsules": capsules}
    elif kind == "channel":
        out |= {"flow": "channel", "nx": _log_int(rng, 96, 320), "ny": _log_int(rng, 40, 160),
                "nz": _log_int(rng, 40, 160), "radius": 6.0, "capsules": False}
    elif kind == "study":
        out |= {"flow": "study", "nx": rng.randint(64, 130), "ny": rng.randint(64, 130), "nz": rng.randint(120, 240),
                "radius": 4.0, "capsules": True}
    else:
        out |= {"flow": "swarm", "nx": _log_int(rng, 128, 448), "ny": _log_int(rng, 120, 256),
                "nz": _log_int(rng, 120, 256), "radius": 4.0, "capsules": rng.random() < 0.6}
    cells = out["nx"] * out["ny"] * out["nz"]
    out["steps"] = max(1, min(steps, int(3e8 / cells) if prec != "f64" else int(7e7 / cells)))
    return out


# ---- what a user's program holds -----------------------------------------------


def _scenario(case, seed):
    """The seeded scenario of a step or gradient case."""
    rng = wl.SplitMix64(0xC0FFEE + 1009 * seed)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    if case["kind"] == "gradient":
        sc = wl.design_swimmer(case["capsules"], seed=seed, steps=case["steps"])
        shift = tuple(0.5 * (n - m) for n, m in zip((nx, ny, nz), (sc.nx, sc.ny, sc.nz)))
        sc.nx, sc.ny, sc.nz = nx, ny, nz
        for b in sc.bodies:
            b.pos = tuple(p + d for p, d in zip(b.pos, shift))
        amp = rng.uniform(0.6, 1.4)
        for d in sc.drives:
            d.amp *= amp
        return sc
    if case["flow"] == "swarm":
        most = max(1, min(8, (nx // 80) * (ny // 80) * (nz // 80)))
        return wl.capsule_swarm(nx, ny, nz, swimmers=most, seed=seed, mix=not case["capsules"])
    if case["flow"] == "study":
        label = rng.choice(("g", "h", "i", "j"))
        sc, _ = design_study.design(label, (nx, ny, nz), period=4000, t_off=(20000, 21000))
        for b in sc.bodies:
            b.pos = tuple(p + rng.uniform(-0.1, 0.1) for p in b.pos)
        return sc
    r = case["radius"]
    centre = tuple((n - 1) / 2.0 for n in (nx, ny, nz))
    amp = rng.uniform(2e-4, 8e-4)
    if case["flow"] == "channel":
        sc = wl.Scenario("channel", nx, ny, nz, 1.0, bc=wl.PERIODIC_X, g=(rng.uniform(1e-7, 2e-7), 0.0, 0.0))
        wl.add_swimmer(sc, centre, (1.0, 0.0, 0.0, 0.0), (wl.SPHERE,) * 3, r, 0.0, 20.0, 0.02, 0.01, amp, 1000.0)
    else:
        sc = wl.Scenario("box", nx, ny, nz, 1.0)
        shape = wl.CAPSULE if case["capsules"] else wl.SPHERE
        half = r * (2 if case["capsules"] else 1)
        wl.add_swimmer(sc, centre, (1.0, 0.0, 0.0, 0.0), (shape,) * 3, r, 2 * r, 2 * half + 4.0, 0.01, 0.005, amp,
                       400.0, density=2.0)
    for b in sc.bodies:
        b.pos = tuple(p + rng.uniform(-0.1, 0.1) for p in b.pos)
    return sc


def _options(case):
    return lbm.OPT_AVERAGE_FORCE if case.get("flow") == "study" else 0


def _members(case, seed):
    """Seeded swimmers in the boxes of the 96-box ensemble (the boxes' sizes
    do not depend on the seed)."""
    boxes = [sc.nx for sc in wl.ensemble_members(96) if sc.nx <= case["edge_max"]]
    boxes = (boxes * math.ceil(case["members"] / len(boxes)))[:case["members"]]
    pool, k = {}, 0
    while any(boxes.count(n) > len(pool.get(n, ())) for n in set(boxes)):
        for sc in wl.ensemble_members(96, seed=seed + 7919 * k):
            pool.setdefault(sc.nx, []).append(sc)
        k += 1
    return [pool[n].pop() for n in boxes]


def _static_arrays(case, seed, device):
    """Populations near rest, a cell map of spheres on a loose grid and body
    states with small velocities, as torch tensors on `device`."""
    rng = np.random.default_rng(seed)
    n = (case["nx"], case["ny"], case["nz"])
    r, pitch = case["radius"], 2 * math.ceil(case["radius"]) + 4
    sites = [(i, j, k) for k in range(n[2] // pitch) for j in range(n[1] // pitch) for i in range(n[0] // pitch)]
    nb = case["bodies"]
    pick = rng.choice(len(sites), nb, replace=False)
    state = np.zeros((nb, 13))
    for b, s in enumerate(pick):
        state[b, :3] = [(sites[s][a] + 0.5) * pitch - 0.5 + rng.uniform(-0.4, 0.4) for a in range(3)]
    state[:, 3] = 1.0
    state[:, 7:13] = rng.uniform(-1e-3, 1e-3, (nb, 6))
    gen = torch.Generator(device="cpu").manual_seed(seed)
    cells = n[0] * n[1] * n[2]
    w = torch.tensor(_W, dtype=torch.float64)
    pop = (w[:, None] * (1.0 + 0.01 * torch.randn(19, cells, generator=gen, dtype=torch.float64))).to(device)
    flags = torch.zeros(n[2], n[1], n[0], dtype=torch.uint8)
    z, y, x = torch.meshgrid(*(torch.arange(v, dtype=torch.float64) for v in (n[2], n[1], n[0])), indexing="ij")
    for b in range(nb):
        d2 = (x - state[b, 0]) ** 2 + (y - state[b, 1]) ** 2 + (z - state[b, 2]) ** 2
        flags[d2 <= r * r] = b + 1
    return pop, flags.to(device).reshape(-1), torch.from_numpy(state).to(device)


_FIELDS = {"u": (("u", lbm.FIELD_U, 3),), "rho_u": (("rho", lbm.FIELD_RHO, 1), ("u", lbm.FIELD_U, 3)),
           "pop": (("pop", lbm.FIELD_POP, 19),)}


def prepare(case, seed):
    if case["kind"] == "static":
        pop, flags, bodies = _static_arrays(case, seed, "cuda")
        out = torch.zeros(case["bodies"], 6, dtype=torch.float64, device="cuda")
        ptr = [ctypes.c_void_p(t.data_ptr()) for t in (pop, flags, bodies)]
        return {"kind": "static", "lib": lbm.load_library(), "out": out, "keep": (pop, flags, bodies),
                "args": (*ptr, case["bodies"], case["nx"], case["ny"], case["nz"], case["bc"], case["half_width"],
                         ctypes.c_void_p(out.data_ptr()))}
    if case["kind"] == "gradient":
        sc = _scenario(case, seed)
        dtype = torch.float64 if case["precision"] == "f64" else torch.float32
        params = {k: v.to(dtype) for k, v in autograd.scenario_parameters(sc).items()}
        return {"kind": "gradient", "sc": sc, "params": params, "case": case}
    if case["kind"] == "ensemble":
        lats = [lbm.from_scenario(sc, precision=case["precision"]) for sc in _members(case, seed)]
        ens = lbm.Ensemble(lats)
        ens.step(case["warm"])
        ens.autotune(3)
        ens.sync()
        sizes = [19 * lat.cells for lat in lats]
        f64 = case["precision"] == "f64"
        flat = torch.empty(sum(sizes), dtype=torch.float64 if f64 else torch.float32, device="cuda")
        return {"kind": "ensemble", "ens": ens, "lats": lats, "flat": flat, "parts": flat.split(sizes),
                "steps": case["steps"], "dtype": lbm.DTYPE_F64 if f64 else lbm.DTYPE_F32}
    sc = _scenario(case, seed)
    lat = lbm.from_scenario(sc, precision=case["precision"], options=_options(case))
    lat.step(1)
    if case["tuned"]:
        lat.autotune(3)
    lat.step(case["warm"] - 1)
    lat.sync()
    f64 = case["precision"] == "f64"
    fields = [(name, what, torch.empty((lead, sc.nz, sc.ny, sc.nx), device="cuda",
                                       dtype=torch.float64 if f64 else torch.float32))
              for name, what, lead in _FIELDS[case["field"]]]
    return {"kind": "step", "lat": lat, "steps": case["steps"], "fields": fields,
            "dtype": lbm.DTYPE_F64 if f64 else lbm.DTYPE_F32}


def run(state):
    if state["kind"] == "static":
        stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
        rc = state["lib"].lbm_momentum_exchange_static(*state["args"], stream)
        if rc != lbm.OK:
            raise lbm.LbmError(rc, "lbm_momentum_exchange_static")
        return state["out"]
    if state["kind"] == "gradient":
        case = state["case"]
        leaf = {k: v.detach().requires_grad_(True) for k, v in state["params"].items()}
        final = autograd.swimmer_run(state["sc"], case["steps"], **leaf, segment=case["segment"],
                                     precision=case["precision"])
        final[:, 0].mean().backward()           # the swimmer's net x displacement
        return {"final": final.detach(), "grad": {k: v.grad for k, v in leaf.items()}}
    if state["kind"] == "ensemble":
        state["ens"].step(state["steps"])
        for lat, part in zip(state["lats"], state["parts"]):
            lat.field_device(lbm.FIELD_POP, part, state["dtype"])
        return {"pop": state["flat"], "bodies": np.stack([lat.bodies() for lat in state["lats"]])}
    lat = state["lat"]
    lat.step(state["steps"])
    out = {}
    for name, what, t in state["fields"]:
        lat.field_device(what, t, state["dtype"])
        out[name] = t
    out["bodies"] = lat.bodies()
    return out


# ---- what a pass cannot do without ----------------------------------------------

_ES = {"f64": 8, "f32": 4, "f16": 2, "bf16": 2}
_FLOPS_CELL = 230           # moments, equilibrium and relaxation of 19 populations


def _cells(case, seed=1):
    if case["kind"] == "ensemble":
        return sum(sc.cells for sc in _members(case, seed))
    return case["nx"] * case["ny"] * case["nz"]


def work(case):
    if case["kind"] == "static":
        shell = 4.0 * math.pi * case["radius"] ** 2            # fluid cells with links, 19 populations each
        side = 2 * case["half_width"] + 1
        return {"bytes": case["bodies"] * (side ** 3 + 152 * shell + 152), "flops": case["bodies"] * shell * 5 * 60}
    C = _cells(case)
    es = _ES[case["precision"]]
    step = (2 * 19 * es + 1) * C
    if case["kind"] == "gradient":
        # the recorded forward, the recomputation from checkpoints and the
        # reverse step: populations and adjoint in, adjoint out, two flag bytes
        return {"bytes": case["steps"] * (2 * step + (3 * 19 * es + 2) * C),
                "flops": case["steps"] * 4 * _FLOPS_CELL * C}
    if case["kind"] == "ensemble":
        return {"bytes": case["steps"] * step + 19 * (es + max(es, 4)) * C, "flops": case["steps"] * _FLOPS_CELL * C}
    lead = sum(f[2] for f in _FIELDS[case["field"]])
    out = (19 * es + lead * (8 if case["precision"] == "f64" else 4)) * C
    return {"bytes": case["steps"] * step + out, "flops": case["steps"] * _FLOPS_CELL * C}


# ---- the method in 64 bits, in plain torch ----------------------------------------

_E = ((0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
      (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1),
      (0, -1, 1))
_W = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
_OPP = [0] + [a + 1 if a % 2 else a - 1 for a in range(1, 19)]


def _rotation(q):
    w, x, y, z = q.unbind(-1)
    return torch.stack((1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)), -1).reshape(-1, 3, 3)


class _Plain:
    """The coupled step on torch tensors in float64: G [19, cells] are the
    post-collision populations, states [bodies, 13] position, quaternion,
    velocity and angular velocity."""

    def __init__(self, sc, averaged, device, params=None):
        t = lambda v: torch.tensor(v, dtype=torch.float64, device=device)
        self.sc, self.averaged, self.device = sc, averaged, device
        self.n = (sc.nx, sc.ny, sc.nz)
        self.periodic = [bool(sc.bc >> a & 1) for a in range(3)]
        self.size = t([float(v) if p else math.inf for v, p in zip(self.n, self.periodic)])
        self.e, self.w = t(_E), t(_W)
        self.ei = torch.tensor(_E, device=device)
        self.opp = torch.tensor(_OPP, device=device)
        self.radius, self.capsule = t([b.radius for b in sc.bodies]), t([float(b.shape) for b in sc.bodies])
        p = params or {"amp": t([d.amp for d in sc.drives]), "phase": t([d.phase for d in sc.drives]),
                       "k": t([s.k for s in sc.springs]), "rest": t([s.rest for s in sc.springs]),
                       "damping": t([s.damping for s in sc.springs]), "mass": t([b.mass for b in sc.bodies]),
                       "length": t([b.length for b in sc.bodies])}
        self.p = p
        self.length = p["length"].detach()
        self.freq, self.off = t([d.freq for d in sc.drives]), t([d.t_off for d in sc.drives])
        self.axis = t([d.axis for d in sc.drives])
        idx = lambda v: torch.tensor(v, dtype=torch.long, device=device)
        self.driven = idx([d.body for d in sc.drives])
        self.si, self.sj = idx([s.i for s in sc.springs]), idx([s.j for s in sc.springs])
        r, l, m = self.radius, p["length"] * self.capsule, p["mass"]
        vc, vh = math.pi * r * r * l, 2 / 3 * math.pi * r ** 3
        self.volume = vc + 2 * vh
        mc, mh = m * vc / self.volume, m * vh / self.volume
        along = 0.5 * mc * r * r + 0.8 * mh * r * r
        across = mc * (r * r / 4 + l * l / 12) + 2 * mh * (0.4 * r * r + l * l / 4 + 3 * l * r / 8)
        self.inertia = torch.stack((along, across, across), -1)
        self.g = t(sc.g)
        self.t = 0
        half = int(max(math.ceil(b.radius + b.length / 2) for b in sc.bodies)) + 4
        a = torch.arange(-half, half + 1, device=device)
        self.cube = torch.stack(torch.meshgrid(a, a, a, indexing="ij"), -1).reshape(-1, 3)

    def start(self, state0=None):
        """Fluid at rest, the bodies at their start."""
        C = self.n[0] * self.n[1] * self.n[2]
        if state0 is None:
            state0 = torch.zeros(len(self.sc.bodies), 13, dtype=torch.float64, device=self.device)
            for k, b in enumerate(self.sc.bodies):
                q = np.asarray(b.orient, dtype=np.float64)
                state0[k, :3] = torch.tensor(b.pos, dtype=torch.float64)
                state0[k, 3:7] = torch.from_numpy(q / np.linalg.norm(q))
        G = self.w[:, None].expand(19, C).contiguous()
        return G, state0, state0, self.map(state0)[0], None

    def offset(self, p, x):
        """p - x, minimum image on the periodic axes."""
        d = p - x
        whole = torch.where(torch.isinf(self.size), 0.0, torch.round(d.detach() / self.size) * self.size)
        return d - torch.nan_to_num(whole)

    def index(self, cell):
        """Linear index of wrapped cells [..., 3] and which lie beyond a wall."""
        beyond = torch.zeros(cell.shape[:-1], dtype=torch.bool, device=self.device)
        parts = []
        for a in range(3):
            v = cell[..., a]
            if not self.periodic[a]:
                beyond = beyond | (v < 0) | (v >= self.n[a])
            parts.append(v % self.n[a])
        return (parts[2] * self.n[1] + parts[1]) * self.n[0] + parts[0], beyond

    def map(self, state):
        """(body of each cell or -1, the cells within reach of a body)."""
        s = state.detach()
        cell = torch.floor(s[:, None, :3]).long() + self.cube
        lin, beyond = self.index(cell)
        d = self.offset(cell.double(), s[:, None, :3])
        ax = _rotation(s[:, 3:7])[:, :, 0]
        h = 0.5 * self.length[:, None]
        along = (d * ax[:, None, :]).sum(-1).clamp(min=-h, max=h) * self.capsule[:, None]
        far = d - along[..., None] * ax[:, None, :]
        inside = ((far * far).sum(-1) <= (self.radius ** 2)[:, None]) & ~beyond
        bid = torch.full((self.n[0] * self.n[1] * self.n[2],), -1, dtype=torch.long, device=self.device)
        who = torch.arange(len(s), device=self.device)[:, None].expand_as(lin)
        bid[lin[inside]] = who[inside]
        near = torch.unique(lin[~beyond])
        x, yz = near % self.n[0], near // self.n[0]
        return bid, torch.stack((x, yz % self.n[1], yz // self.n[1]), -1)

    def wall_velocity(self, state, body, point):
        s = state[body]
        return s[..., 7:10] + torch.linalg.cross(s[..., 10:13], self.offset(point, s[..., :3]))

    def collide(self, F, solid):
        tau, g, forced = self.sc.tau, self.sc.g, any(self.sc.g)
        rho = F.sum(0)
        u = []
        for a in range(3):
            plus = sum(F[b] for b in range(19) if _E[b][a] > 0)
            u.append((plus - sum(F[b] for b in range(19) if _E[b][a] < 0) + 0.5 * g[a]) / rho)
        uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2]
        ug = u[0] * g[0] + u[1] * g[1] + u[2] * g[2] if forced else None
        out = []
        for b in range(19):
            eu = sum(_E[b][a] * u[a] for a in range(3) if _E[b][a]) if b else 0.0 * rho
            post = F[b] - (F[b] - _W[b] * rho * (1 + 3 * eu + 4.5 * eu * eu - 1.5 * uu)) / tau
            if forced:
                eg = sum(_E[b][a] * g[a] for a in range(3))
                post = post + (1 - 0.5 / tau) * _W[b] * (3 * (eg - ug) + 9 * eu * eg)
            out.append(torch.where(solid, _W[b], post))
        return torch.stack(out)

    def step(self, G, prev, cur, bid_prev, load_prev):
        """One coupled step: (G, states n-1, n, map of n-1, load of n-1) ->
        the same one step on."""
        nx, ny, nz = self.n
        bid, near = self.map(cur)
        at, _ = self.index(near)
        F = torch.stack([torch.roll(G[b].view(nz, ny, nx), (e[2], e[1], e[0]), (0, 1, 2)) for b, e in enumerate(_E)])
        for b, e in enumerate(_E):
            for a in range(3):
                if e[a] and not self.periodic[a]:               # halfway bounce-back at the walls
                    face = [slice(None)] * 3
                    face[2 - a] = 0 if e[a] > 0 else self.n[a] - 1
                    F[(b, *face)] = G[_OPP[b]].view(nz, ny, nx)[tuple(face)]
        F = F.view(19, -1)
        # moving bounce-back: sources x - e that were solid
        src, beyond = self.index(near[None] - self.ei[:, None])
        hit = (bid_prev[src] >= 0) & ~beyond & (bid_prev[at] < 0)[None] & (self.e != 0).any(-1)[:, None]
        b, i = hit.nonzero(as_tuple=True)
        if len(b):
            c, y = at[i], near[i].double() - self.e[b]
            uw = self.wall_velocity(prev, bid_prev[src[b, i]], y)
            val = G[self.opp[b], c] + 6 * self.w[b] * G[:, c].sum(0) * (self.e[b] * uw).sum(-1)
            F = F.index_put((b, c), val) if F.requires_grad else F.index_put_((b, c), val)
        # uncovered cells: equilibrium at the mean density of the neighbours
        bare = ((bid_prev[at] >= 0) & (bid[at] < 0)).nonzero()[:, 0]
        if len(bare):
            c, p = at[bare], near[bare]
            nb, out = self.index(p[None] + self.ei[1:, None])
            ok = (~out & (bid_prev[nb] < 0) & (bid[nb] < 0)).double()
            cnt = ok.sum(0)
            mean = torch.where(cnt > 0, (G[:, nb].sum(0) * ok).sum(0) / cnt.clamp(min=1), 1.0)
            uw = self.wall_velocity(cur, bid_prev[c], p.double())
            eu, uu = self.e @ uw.T, (uw * uw).sum(-1)
            feq = self.w[:, None] * mean * (1 + 3 * eu + 4.5 * eu * eu - 1.5 * uu)
            a = torch.arange(19, device=self.device)[:, None].expand(-1, len(c))
            F = F.index_put((a, c[None].expand(19, -1)), feq)
        G = self.collide(F, bid >= 0)
        # momentum exchange over the links of the new map
        dst, beyond = self.index(near[None] + self.ei[:, None])
        hit = (bid[dst] >= 0) & ~beyond & (bid[at] < 0)[None]
        b, i = hit.nonzero(as_tuple=True)
        c, k = at[i], bid[dst[b, i]]
        uw = self.wall_velocity(cur, k, near[i].double() + self.e[b])
        mag = 2 * G[b, c] - 6 * self.w[b] * G[:, c].sum(0) * (self.e[b] * uw).sum(-1)
        link = self.e[b] * mag[:, None]
        arm = self.offset(near[i].double() + 0.5 * self.e[b], cur[k][:, :3])
        both = torch.cat((link, torch.linalg.cross(arm, link)), -1)
        load = torch.zeros(len(cur), 6, dtype=torch.float64, device=self.device).index_add(0, k, both)
        nxt = self.integrate(cur, load if load_prev is None or not self.averaged else 0.5 * (load + load_prev))
        self.t += 1
        return G, cur, nxt, bid, load

    def integrate(self, s, load):
        p, t = self.p, self.t
        R = _rotation(s[:, 3:7])
        F = load[:, :3] + self.g * self.volume[:, None]
        omega = 2 * math.pi * self.freq
        on = (t >= (p["phase"] / omega).detach()) & (t < self.off)
        f = torch.where(on, p["amp"] * torch.sin(omega * t - p["phase"]), 0.0)
        F = F.index_add(0, self.driven, f[:, None] * (R[self.driven] @ self.axis[..., None])[..., 0])
        d = s[self.si, :3] - s[self.sj, :3]
        length = d.norm(dim=-1, keepdim=True)
        fs = -p["k"][:, None] * (length - p["rest"][:, None]) * d / length \
            - p["damping"][:, None] * (s[self.si, 7:10] - s[self.sj, 7:10])
        F = F.index_add(0, self.si, fs).index_add(0, self.sj, -fs)
        V = s[:, 7:10] + F / p["mass"][:, None]
        X = s[:, :3] + V
        body = (R.transpose(1, 2) @ load[:, 3:, None])[..., 0] / self.inertia
        W = s[:, 10:13] + (R @ body[..., None])[..., 0]
        w, v = s[:, 3:4], s[:, 4:7]
        q = torch.cat((w - 0.5 * (W * v).sum(-1, keepdim=True), v + 0.5 * (w * W + torch.linalg.cross(W, v))), -1)
        return torch.cat((X, q / q.norm(dim=-1, keepdim=True), V, W), -1)

    def moments(self, G):
        """Density and velocity of the last step's map (1 and 0 in obstacles)."""
        rho = G.sum(0)
        u = torch.stack([(sum(_E[b][a] * G[b] for b in range(19) if _E[b][a]) - 0.5 * self.sc.g[a]) / rho
                         for a in range(3)])
        return rho, u


def _run_plain(sc, averaged, steps, device):
    sim = _Plain(sc, averaged, device)
    s = sim.start()
    with torch.no_grad():
        for _ in range(steps):
            s = sim.step(*s)
    return sim, s


def _exact_gradient(case, seed, device):
    from torch.utils.checkpoint import checkpoint
    sc = _scenario(case, seed)
    given = autograd.scenario_parameters(sc)
    if case["precision"] != "f64":
        given = {k: v.float() for k, v in given.items()}
    leaf = {k: v.double().to(device) for k, v in given.items()}
    q = leaf["state0"][:, 3:7]
    leaf["state0"][:, 3:7] = q / q.norm(dim=-1, keepdim=True)
    for v in leaf.values():
        v.requires_grad_(True)
    sim = _Plain(sc, False, device, {k: v for k, v in leaf.items() if k != "state0"})

    def block(t, n, *s):
        sim.t = t
        for _ in range(n):
            s = sim.step(*s[:4], None)
        return s[:4]

    s, t = sim.start(leaf["state0"])[:4], 0
    while t < case["steps"]:
        n = min(16, case["steps"] - t)
        s, t = checkpoint(block, t, n, *s, use_reentrant=False), t + n
    s[2][:, 0].mean().backward()
    return {"final": s[2].detach(), "grad": {k: v.grad for k, v in leaf.items()}}


def exact(case, seed):
    device = "cuda" if torch.cuda.is_available() else "cpu"
    if case["kind"] == "static":
        pop, flags, state = _static_arrays(case, seed, device)
        sc = wl.Scenario("static", case["nx"], case["ny"], case["nz"], 1.0, bc=case["bc"])
        sc.bodies = [wl.Body(wl.SPHERE, case["radius"], 0.0, 1.0, (0.0, 0.0, 0.0)) for _ in range(case["bodies"])]
        sim = _Plain(sc, False, device)
        bid = flags.long() - 1
        _, near = sim.map(state)
        at, _ = sim.index(near)
        dst, beyond = sim.index(near[None] + sim.ei[:, None])
        b, i = ((bid[dst] >= 0) & ~beyond & (bid[at] < 0)[None]).nonzero(as_tuple=True)
        c, k = at[i], bid[dst[b, i]]
        uw = sim.wall_velocity(state, k, near[i].double() + sim.e[b])
        link = sim.e[b] * (2 * pop[b, c] - 6 * sim.w[b] * pop[:, c].sum(0) * (sim.e[b] * uw).sum(-1))[:, None]
        arm = sim.offset(near[i].double() + 0.5 * sim.e[b], state[k][:, :3])
        both = torch.cat((link, torch.linalg.cross(arm, link)), -1)
        return torch.zeros(case["bodies"], 6, dtype=torch.float64, device=device).index_add(0, k, both)
    if case["kind"] == "gradient":
        return _exact_gradient(case, seed, device)
    if case["kind"] == "ensemble":
        pop, bodies = [], []
        for sc in _members(case, seed):
            _, s = _run_plain(sc, False, case["warm"] + case["steps"], device)
            pop.append(s[0].reshape(-1))
            bodies.append(s[2].cpu().numpy())
        return {"pop": torch.cat(pop), "bodies": np.stack(bodies)}
    sc = _scenario(case, seed)
    sim, (G, _, state, bid, _) = _run_plain(sc, bool(_options(case)), case["warm"] + case["steps"], device)
    shape = (-1, sc.nz, sc.ny, sc.nx)
    if case["field"] == "pop":
        out = {"pop": G.view(shape)}
    else:
        rho, u = sim.moments(G)
        out = {"u": torch.where(bid >= 0, 0.0, u).view(shape)}
        if case["field"] == "rho_u":
            out["rho"] = torch.where(bid >= 0, 1.0, rho).view(shape)
    out["bodies"] = state.cpu().numpy()
    return out
