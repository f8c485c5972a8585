"""The work that users of the library have it do, as measurable cases.

A case is a dict of plain values.  Its `kind` names the call it makes:

  step      Context.step: one Lagrangian step with the previous footprint cleared
  graph     StepGraph.launch: a captured pair of steps, replayed
  host      Context.step_host: the step with the body state in page-locked memory
  pc        Context.step_pc: one strong-coupling (Hamming) step
  transfer  Context.interpolate, then Context.spread of the marker forces
  forces    Context.compute_forces
  rollout   autograd.rollout: forward and backward through several steps
  flow      Flow.step without bodies: the fluid phase alone
  coupled   Flow.step with bodies: the loosely coupled step

`bodies` names the scene: equal drops in a random flow, closed bodies of uneven
size, or a closed membrane around two clamped leaflets (two-sided probes,
van Gelder springs).  Sizes are those of the library's benchmark and tests, or
lie between them.  `exact` restates the method in plain torch float64 from its
definitions (general 4x4 moment systems, energies differentiated by autograd,
transforms in float64) and shares nothing with the library.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1612_03399_gb300 import workloads as W

KINDS = ("step", "graph", "host", "pc", "transfer", "forces", "rollout", "flow", "coupled")
ALPHA = 0.3
GAMMA = (8.0 / 15.0, 5.0 / 12.0, 3.0 / 4.0)
RHO = (0.0, -17.0 / 60.0, -5.0 / 12.0)


def _case(name, kind, bodies, count, level, nx, ny, nz, **options):
    c = {"kind": kind, "bodies": bodies, "count": count, "level": level, "nx": nx, "ny": ny,
         "nz": nz, "variant": 1, "pressure": False, "steps": 1, "nu": 0.0}
    c.update(options)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: one 1280-face drop in shear, launch and latency bound
        _case("step_one_drop", "step", "drops", 1, 3, 64, 64, 64),
        # the library's headline: 1000 drops of 1280 faces on 512^3
        _case("step_1000_drops", "step", "drops", 1000, 3, 512, 512, 512),
        # bodies of 320 to 20480 faces, on a grid whose rows are not whole float4s
        _case("step_uneven", "step", "uneven", 128, 5, 301, 288, 310),
        # a finely meshed membrane with leaflets under pressure: many faces per cell
        _case("step_membrane", "step", "membrane", 3, 7, 256, 256, 256, pressure=True),
        # reproducible fields: the tile-owned spread
        _case("step_reproducible", "step", "drops", 250, 3, 256, 256, 256, variant=2),
        # a captured pair of steps, the way a long frozen-flow run is driven
        _case("graph_100_drops", "graph", "drops", 100, 3, 192, 192, 192),
        # the state held by a host program: copies in and out with every step
        _case("host_500_drops", "host", "drops", 500, 3, 320, 320, 320),
        # strong coupling
        _case("pc_200_drops", "pc", "drops", 200, 3, 256, 256, 256),
        # the transfer pair alone, on a ragged box, with pressure loads
        _case("transfer_uneven", "transfer", "uneven", 48, 4, 150, 162, 140, pressure=True),
        # calibration: forward and backward through steps of 2562-node drops
        _case("rollout_48_drops", "rollout", "drops", 48, 4, 160, 160, 160, steps=4),
        # the fluid phase alone on a ragged box, viscous enough for the Fourier solve
        _case("flow_ragged", "flow", "none", 0, 0, 200, 180, 144, nu=0.5),
        # the coupled benchmark: 1000 drops in a solved flow on 256^3
        _case("coupled_1000_drops", "coupled", "drops", 1000, 3, 256, 256, 256, nu=0.01),
    ]


def draw(rng):
    kind = rng.choice(KINDS + ("step", "step", "coupled"))
    log = lambda a, b: int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))
    base = log(48, 220 if kind in ("flow", "coupled") else 300)
    n = [max(24, int(base * rng.uniform(0.85, 1.15))) for _ in range(3)]
    if rng.random() < 0.6:                       # whole float4 rows are the usual choice
        n[0] = max(24, n[0] // 4 * 4)
    cells = n[0] * n[1] * n[2]
    if kind == "flow":
        return _case("", kind, "none", 0, 0, *n, nu=rng.choice((0.002, 0.01, 0.05, 0.5)))
    scene = "drops" if kind in ("rollout", "coupled", "graph") else rng.choice(
        ("drops", "drops", "uneven", "membrane"))
    # no denser than the benchmark's 1000 drops on 256^3
    most = max(1, cells // 16800)
    if scene == "drops":
        # the coupled forcing wants faces below two cells: the level follows the drop's size
        count, level = min(log(1, 800), most), 3
        if kind in ("rollout", "coupled"):
            r = 0.3 * min(n) / max(1, math.ceil(count ** (1 / 3)))
            level = 3 if r < 16 else (4 if r < 32 else 5)
        if kind == "rollout":
            count = min(count, 48 if level <= 4 else 8)
    elif scene == "uneven":
        count, level = min(log(2, 128), max(2, most // 4)), rng.choice((3, 4, 5))
    else:
        count, level = 3, (5 if min(n) < 100 else 6)
    return _case("", kind, scene, count, level, *n,
                 variant=rng.choice((1, 1, 1, 2)) if kind in ("step", "transfer", "pc") else 1,
                 pressure=kind in ("step", "transfer") and rng.random() < 0.4,
                 steps=rng.choice((2, 3, 4)) if kind == "rollout" else 1,
                 nu=rng.choice((0.005, 0.01, 0.02)) if kind == "coupled" else 0.0)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------


def _grid(case):
    n = (case["nx"], case["ny"], case["nz"])
    m = max(n)
    return W.Grid(n, tuple(k / m for k in n))    # cubic cells


@functools.lru_cache(maxsize=4)
def _leaflet(faces):
    return W.elliptic_sheet(0.12, 0.08, faces, np.random.default_rng(4), jitter=0.1)


def _scene(case, rng):
    """Bodies: drops and uneven bodies on a jittered lattice (no two overlap),
    or the membrane with its leaflets."""
    grid = _grid(case)
    L = np.array(grid.L)
    if case["bodies"] == "none":
        return []
    if case["bodies"] == "membrane":
        v, t = W.icosphere(case["level"])
        c = L / 2
        out = [W.Body(rest=c + v * (L * np.array([0.3, 0.3, 0.45])), tri=t, origin=c.copy(), ks=10.0,
                      kb=0.1, level=case["level"], spring_model=1)]
        for dz in (-0.1, 0.1):
            sv, st, rim = _leaflet(len(t) // 13)
            o = c + np.array([0.0, 0.0, dz * L[2]])
            out.append(W.Body(rest=o + sv * min(L), tri=st, origin=o, closed=False, clamped=rim,
                              ks=10.0, kb=1.0, ka=1.0, kA=0.0, kv=0.0, spring_model=1))
        return out
    nb = case["count"]
    m = max(1, math.ceil(nb ** (1 / 3)))
    site = rng.permutation(m ** 3)[:nb]
    at = np.stack([site % m, site // m % m, site // (m * m)], 1)
    pitch = L.min() / m
    out = []
    for i in range(nb):
        if case["bodies"] == "drops":
            level, r, stretch = case["level"], pitch * rng.uniform(0.15, 0.3), np.ones(3)
        else:
            level = 2 + _level_of(i, case)
            r = 0.26 * pitch * 2.0 ** (level - case["level"])
            stretch = rng.uniform(1.0, 1.5, 3)
        v, t = W.icosphere(level)
        rot = W.random_rotation(rng)
        c = (at[i] + 0.5 + rng.uniform(-0.1, 0.1, 3)) * L / m
        out.append(W.Body(rest=c + r * (((v @ rot) * stretch) @ rot.T), tri=t, origin=c, level=level,
                          ks=rng.uniform(0.5, 2.0), kb=rng.uniform(0.005, 0.02)))
    return out


def _level_share(k):
    p = np.array([0.4, 0.3, 0.2, 0.1][:k])
    return p / p.sum()


def _level_of(i, case):
    """Body i's size class: the same for every seed, shares 0.4, 0.3, 0.2, 0.1."""
    edges = np.cumsum(_level_share(case["level"] - 1))
    return int(np.searchsorted(edges, (i + 0.5) / case["count"]))


class Inputs:
    """What a user's program holds before the call, without the library's handles."""

    def __init__(self, case, seed):
        rng = np.random.default_rng([seed, 1612])
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.grid = _grid(case)
        self.bodies = _scene(case, rng)
        n = self.grid.n
        # small steps where a pass carries on from the last one: the bodies keep their shape
        self.dt = 1e-4 if case["bodies"] == "membrane" or case["kind"] in ("graph", "pc") else 1e-3
        self.mu = case["nu"] if case["kind"] == "coupled" else 1.0
        spec = W.fourier_modes(32, 8 if min(n) >= 64 else 3, 1.0, rng)
        if case["count"] == 1 and case["kind"] in ("step", "graph", "host", "pc", "rollout"):
            spec = {"kind": "shear"}
        self.fields = W.sample_field(spec, self.grid, device=dev)
        self.p = None
        if case["pressure"]:
            self.p = W.sample_pressure(W.pressure_modes(32, 8 if min(n) >= 64 else 3, 1.0, rng),
                                       self.grid, device=dev)
        if case["kind"] in ("flow", "coupled"):
            rate = sum(float(f.abs().max()) / h for f, h in zip(self.fields, self.grid.h))
            self.dt = 0.5 / rate                  # CFL 0.5
            self.p = torch.zeros_like(self.fields[0])
        x, v = [], []
        for b in self.bodies:
            e = np.linalg.norm(b.rest[b.tri[:64, 1]] - b.rest[b.tri[:64, 0]], axis=1).mean()
            d = 0.02 * e * rng.standard_normal(b.rest.shape)
            rel = (b.rest - b.origin) * (1.0 + 0.02 * rng.standard_normal(3))
            drift = 0.2 * rng.standard_normal(3) + 0.02 * e * rng.standard_normal(b.rest.shape)
            if b.clamped is not None:
                d[b.clamped], drift[b.clamped] = 0.0, 0.0
                rel[b.clamped] = (b.rest - b.origin)[b.clamped]
            x.append(rel + d)
            v.append(drift)
        to = lambda a: torch.tensor(np.ascontiguousarray(np.concatenate(a).T.astype(np.float32)),
                                    device=dev)
        self.x, self.v, self.accel = (to(x), to(v), None) if x else (None, None, None)
        if case["kind"] == "coupled":
            self.v.zero_()
        if case["pressure"]:
            self.accel = to([rng.standard_normal(a.shape) for a in x])
        self.cot = None
        if case["kind"] == "rollout":
            self.cot = tuple(torch.tensor(rng.standard_normal(tuple(self.x.shape)).astype(np.float32),
                                          device=dev) for _ in range(2))
            self.k = torch.tensor([[b.ks, b.kb, b.ka, b.kA, b.kv] for b in self.bodies],
                                  dtype=torch.float32)


class State:
    pass


def prepare(case, seed):
    from paper_1612_03399_gb300 import _lib
    from paper_1612_03399_gb300 import autograd as A
    i = Inputs(case, seed)
    s = State()
    s.case, s.inputs, s.kind = case, i, case["kind"]
    if s.kind == "rollout":
        s.sim = A.Simulation(i.bodies, i.grid, {"kind": "uniform", "U": (0.0, 0.0, 0.0)}, dt=i.dt,
                             mu=i.mu, alpha=ALPHA)
        for mine, theirs in zip(s.sim.fields, i.fields):
            mine.copy_(theirs)
        return s
    if s.kind in ("flow", "coupled"):
        s.flow = _lib.Flow(i.grid, nu=case["nu"], dt=i.dt)
        s.fields = tuple(f.clone() for f in i.fields)
        s.p = i.p.clone()
    if not i.bodies:
        return s
    s.ctx = _lib.Context(i.bodies, i.grid, dt=i.dt, mu=i.mu, alpha=ALPHA,
                         spread_variant=case["variant"])
    n = i.grid.n
    s.f = tuple(torch.zeros((n[2], n[1], n[0]), device=i.x.device) for _ in range(3))
    if s.kind == "host":
        pin = lambda t: t.cpu().pin_memory()
        s.x, s.v = pin(i.x), pin(i.v)
        s.x1, s.v1 = pin(torch.zeros_like(i.x)), pin(torch.zeros_like(i.x))
    else:
        s.x, s.v = i.x.clone(), i.v.clone()
        s.x1, s.v1 = torch.empty_like(i.x), torch.empty_like(i.x)
    if s.kind == "graph":
        s.graph = s.ctx.graph(s.x, s.v, s.x1, s.v1, i.fields, s.f, 2)
    return s


def run(s):
    i, kind = s.inputs, s.kind
    if kind == "step":
        s.ctx.step(s.x, s.v, i.fields, s.x1, s.v1, s.f, p=i.p, accel=i.accel)
        return _moved(s)
    if kind == "host":
        s.ctx.step_host(s.x, s.v, i.fields, s.x1, s.v1, s.f)
        return _moved(s)
    if kind == "graph":
        s.graph.launch()
        return {"x": s.x, "v": s.v, "f": list(s.f)}
    if kind == "pc":
        s.ctx.step_pc(s.x, s.v, i.fields, s.x1, s.v1, s.f)
        s.x, s.v, s.x1, s.v1 = s.x1, s.v1, s.x, s.v
        return {"x": s.x, "v": s.v, "f": list(s.f)}
    if kind == "transfer":
        U, Fm, Fe = s.ctx.interpolate(s.x, s.v, i.fields, p=i.p, accel=i.accel)
        for f in s.f:
            f.zero_()
        s.ctx.spread(s.x, Fm, s.f)
        return {"U": U, "F_marker": Fm, "F_ext": Fe, "f": list(s.f)}
    if kind == "forces":
        return {"F": s.ctx.compute_forces(s.x, out=s.x1)}
    if kind == "rollout":
        from paper_1612_03399_gb300 import autograd as A
        x, v, k = (t.detach().clone().requires_grad_() for t in (i.x, i.v, i.k))
        xn, vn = A.rollout(s.sim, x, v, k, s.case["steps"], 2)
        gx, gv, gk = torch.autograd.grad((xn, vn), (x, v, k), i.cot)
        return {"x": xn.detach(), "v": vn.detach(), "gx": gx, "gv": gv, "gk": gk}
    if kind == "flow":
        s.flow.step(s.fields, s.p)
        return {"u": list(s.fields), "p": s.p}
    s.flow.step(s.fields, s.p, ctx=s.ctx, x=s.x, v=s.v, x_out=s.x1, v_out=s.v1, f=s.f)
    s.x, s.v, s.x1, s.v1 = s.x1, s.v1, s.x, s.v
    return {"u": list(s.fields), "p": s.p, "x": s.x, "v": s.v, "f": list(s.f)}


def _moved(s):
    return {"x": s.x1, "v": s.v1, "f": list(s.f)}


# ---------------------------------------------------------------------------
# the work of one pass
# ---------------------------------------------------------------------------


def _sizes(case):
    """(vertices, faces, surface in cells) of the scene, the surface at the mean radius."""
    n = (case["nx"], case["ny"], case["nz"])
    if case["bodies"] == "none":
        return 0, 0, 0.0
    if case["bodies"] == "membrane":
        F = int(20 * 4 ** case["level"] * (1 + 2 / 13))
        a, c = 0.3 * min(n), 0.45 * min(n)
        return F // 2, F, 4 * math.pi * (a * a + 2 * a * c) / 3 + 2 * math.pi * 0.0096 * min(n) ** 2
    nb = case["count"]
    pitch = min(n) / max(1, math.ceil(nb ** (1 / 3)))
    if case["bodies"] == "drops":
        F = nb * 20 * 4 ** case["level"]
        return F // 2 + 2 * nb, F, nb * 4 * math.pi * 0.0525 * pitch ** 2
    js = [_level_of(i, case) for i in range(nb)]
    F = sum(20 * 4 ** (2 + j) for j in js)
    S = sum(4 * math.pi * (1.25 * 0.26 * pitch * 2.0 ** (j + 2 - case["level"])) ** 2 for j in js)
    return F // 2 + 2 * nb, F, S


def work(case):
    """Bytes: the state and rest data once, and per velocity (force) component
    the grid nodes that the supports touch, about 5.1 (3.9) per cell of surface;
    flops: the shape functions with their contractions per face, the potentials
    per vertex."""
    V, F, S = _sizes(case)
    N = case["nx"] * case["ny"] * case["nz"]
    lattices = 4 if case["pressure"] else 3
    read = 4 * lattices * min(5.1 * S, 54 * F, N)
    read_c = 12 * min(3.9 * S, 27 * F, N)
    write = 12 * min(3.9 * S, 27 * F, N)
    state, rest = 48 * V, 44 * V
    forces = 900 * V
    kind = case["kind"]
    step = {"bytes": state + rest + read + write, "flops": 1500 * F + forces}
    fluid = {"bytes": 3 * 4 * N * 24, "flops": 3 * N * (200 + 5 * math.log2(max(N, 2)))}
    if kind in ("step", "host"):
        return step
    if kind == "graph":
        return {k: 2 * v for k, v in step.items()}
    if kind == "pc":       # two evaluations of the loads and forces, one spread
        return {"bytes": 2 * (rest + read) + write + 150 * V, "flops": 2500 * F + 2 * forces}
    if kind == "transfer":
        return {"bytes": 24 * V + 36 * F + read + write + 12 * N, "flops": 1500 * F}
    if kind == "forces":
        return {"bytes": 24 * V + rest, "flops": forces}
    if kind == "rollout":  # each state forward, recomputed in part, and backward
        m = case["steps"]
        return {"bytes": m * (2 * step["bytes"] + 48 * V + rest + read),
                "flops": m * (2 * step["flops"] + 4000 * F + 3 * forces)}
    if kind == "flow":
        return fluid
    return {"bytes": fluid["bytes"] + 3 * (read_c + write) + state + rest + read,
            "flops": fluid["flops"] + 3 * 900 * F + 800 * F + forces}


# ---------------------------------------------------------------------------
# the method in float64, from its definitions
# ---------------------------------------------------------------------------

OFFSETS = ((0.0, 0.5, 0.5), (0.5, 0.0, 0.5), (0.5, 0.5, 0.0), (0.5, 0.5, 0.5))
CHUNK = 1 << 17


class Exact:
    def __init__(self, case, seed):
        i = self.i = Inputs(case, seed)
        self.dev = i.fields[0].device
        t = lambda a, dt=torch.float64: torch.as_tensor(np.ascontiguousarray(a), dtype=dt,
                                                        device=self.dev)
        self.n, self.h = i.grid.n, i.grid.h
        self.hv = t(np.array(self.h))
        self.dt, self.mu = i.dt, i.mu
        self.probe = sum(self.h) / 3
        self.kappa = 1.0 / (1.5 * ALPHA) ** 2
        s = np.array([(x, y, z) for z in (-1, 0, 1) for y in (-1, 0, 1) for x in (-1, 0, 1)], float)
        self.S = t(s)
        pk = np.concatenate([np.ones((27, 1)), s], 1)
        self.pk, self.pp = t(pk), t(pk[:, :, None] * pk[:, None, :]).reshape(27, 16)
        if not i.bodies:
            return
        tri, edge, owner_v, vo = [], [], [], 0
        for j, b in enumerate(i.bodies):
            tri.append(b.tri.astype(np.int64) + vo)
            edge.append(_edges(b.tri) + vo)
            owner_v.append(np.full(len(b.rest), j))
            vo += len(b.rest)
        self.V, self.B = vo, len(i.bodies)
        self.owner = t(np.concatenate(owner_v), torch.long)
        self.tri = t(np.concatenate(tri), torch.long)
        e = np.concatenate(edge)
        self.edge = t(e[:, :2], torch.long)
        self.hinge = t(e[e[:, 3] >= 0], torch.long)
        self.fb, self.eb = self.owner[self.tri[:, 0]], self.owner[self.edge[:, 0]]
        self.origin = t(np.array([b.origin for b in i.bodies]))
        self.closed = t(np.array([b.closed for b in i.bodies]), torch.bool)
        self.clamped = t(np.concatenate([np.zeros(len(b.rest), bool) if b.clamped is None else b.clamped
                                         for b in i.bodies]), torch.bool)
        self.mass = t(np.array([b.mass for b in i.bodies]))
        self.k = t(np.array([[b.ks, b.kb, b.ka, b.kA, b.kv if b.closed else 0.0] for b in i.bodies]))
        rest = t(np.concatenate([b.rest - b.origin for b in i.bodies]))
        self.l0 = (rest[self.edge[:, 1]] - rest[self.edge[:, 0]]).norm(dim=1)
        self.c0, self.s0 = self.angle(rest)
        self.A0f = self.normals(rest).norm(dim=1) / 2
        self.A0 = self.per_body(self.A0f)
        self.V0 = torch.where(self.closed, self.volume(rest), 1.0)
        self.m_e = torch.ones_like(self.l0)
        if any(b.spring_model for b in i.bodies):       # van Gelder
            lo = torch.minimum(self.edge[:, 0], self.edge[:, 1]) * self.V + self.edge.max(1).values
            order = torch.argsort(lo)
            acc = torch.zeros_like(self.l0)
            for k in range(3):
                a, b = self.tri[:, k], self.tri[:, (k + 1) % 3]
                at = order[torch.searchsorted(lo[order], torch.minimum(a, b) * self.V + torch.maximum(a, b))]
                acc.index_add_(0, at, self.A0f)
            self.m_e = acc / self.l0 ** 2

    # geometry and potentials (x: [V, 3], body frame)
    def normals(self, x):
        a, b, c = (x[self.tri[:, k]] for k in range(3))
        return torch.linalg.cross(b - a, c - a)

    def per_body(self, q):
        return torch.zeros(self.B, dtype=q.dtype, device=self.dev).index_add(0, self.fb, q)

    def volume(self, x):
        a, b, c = (x[self.tri[:, k]] for k in range(3))
        return self.per_body((a * torch.linalg.cross(b, c)).sum(1) / 6)

    def angle(self, x):
        a, b, c, d = (x[self.hinge[:, k]] for k in range(4))
        n1 = torch.linalg.cross(b - a, c - a)
        n2 = torch.linalg.cross(a - b, d - b)
        n1, n2, e = (q / q.norm(dim=1, keepdim=True) for q in (n1, n2, b - a))
        return (n1 * n2).sum(1), (torch.linalg.cross(n1, n2) * e).sum(1)

    def energy(self, x, k):
        l = (x[self.edge[:, 1]] - x[self.edge[:, 0]]).norm(dim=1)
        w = (0.5 * k[self.eb, 0] * self.m_e * (l - self.l0) ** 2).sum()
        c, s = self.angle(x)
        w = w + (k[self.owner[self.hinge[:, 0]], 1] * (1 - (c * self.c0 + s * self.s0))).sum()
        A = self.normals(x).norm(dim=1) / 2
        w = w + (0.5 * k[self.fb, 2] * (A - self.A0f) ** 2 / self.A0f).sum()
        w = w + (0.5 * k[:, 3] * (self.per_body(A) - self.A0) ** 2 / self.A0).sum()
        vol = 0.5 * k[:, 4] * (self.volume(x) - self.V0) ** 2 / self.V0
        return w + torch.where(self.closed, vol, torch.zeros_like(vol)).sum()

    def internal(self, x, k, graph=False):
        y = x if x.requires_grad else x.detach().requires_grad_()
        with torch.enable_grad():
            return -torch.autograd.grad(self.energy(y, k), y, create_graph=graph)[0]

    # moving least squares at tau (cells)
    def support(self, tau, comp):
        u = tau - torch.tensor(OFFSETS[comp], dtype=tau.dtype, device=self.dev)
        c = torch.floor(u.detach() + 0.5)
        tp = u - c
        delta = self.S[None] - tp[:, None]
        w = torch.exp(-self.kappa * (delta * delta).sum(2))
        at = c.long()[:, None] + self.S.long()[None]
        n = torch.tensor(self.n, device=self.dev)
        at = torch.remainder(at, n)
        return (at[..., 2] * self.n[1] + at[..., 1]) * self.n[0] + at[..., 0], tp, delta, w

    def moments(self, w):
        return (w @ self.pp).reshape(-1, 4, 4)

    def value(self, field, tau, comp):
        at, tp, _, w = self.support(tau, comp)
        c = torch.linalg.solve(self.moments(w), (w * field.reshape(-1)[at].double()) @ self.pk)
        return c[:, 0] + (c[:, 1:] * tp).sum(1)

    def gradient(self, field, tau, comp):
        at, tp, delta, w = self.support(tau, comp)
        q = field.reshape(-1)[at].double()
        M = self.moments(w)
        c = torch.linalg.solve(M, (w * q) @ self.pk)
        r = torch.linalg.solve(M, torch.cat([torch.ones_like(tp[:, :1]), tp], 1))
        out = []
        for e in range(3):
            dw = 2 * self.kappa * delta[..., e] * w
            rhs = (dw * q) @ self.pk - (self.moments(dw) @ c[..., None])[..., 0]
            out.append(c[:, e + 1] + (r * rhs).sum(1))
        return torch.stack(out, 1) / self.hv

    def shape(self, tau, comp):
        at, tp, _, w = self.support(tau, comp)
        r = torch.linalg.solve(self.moments(w), torch.cat([torch.ones_like(tp[:, :1]), tp], 1))
        return at, w * (r @ self.pk.T)

    # per-marker quantities over blocks of faces
    def markers(self, x, v, fields, p=None, accel=None, interp=True, probe=True):
        U, T, A, tau = [], [], [], []
        for o in range(0, len(self.tri), CHUNK):
            tri, fb = self.tri[o:o + CHUNK], self.fb[o:o + CHUNK]
            a, b, c = (x[tri[:, k]] for k in range(3))
            N = torch.linalg.cross(b - a, c - a)
            nn = N.norm(dim=1, keepdim=True)
            n, area = N / nn, nn[:, 0] / 2
            cen = (a + b + c) / 3 + self.origin[fb]
            t = cen / self.hv
            A.append(area)
            tau.append(t)
            if interp:
                U.append(torch.stack([self.value(fields[i], t, i) for i in range(3)], 1))
            if probe:
                two = ~self.closed[fb][:, None]
                load = 0.0
                for side in (1.0, -1.0):
                    if side < 0 and not bool(two.any()):
                        continue
                    on = torch.ones_like(area) if side > 0 else two[:, 0].to(area.dtype)
                    e = (cen + side * self.probe * n) / self.hv
                    G = torch.stack([self.gradient(fields[i], e, i) for i in range(3)], 1)
                    f = self.mu * side * ((G + G.transpose(1, 2)) @ n[..., None])[..., 0]
                    if p is not None:
                        ps = side * self.value(p, e, 3)
                        if accel is not None:
                            am = (accel[tri[:, 0]] + accel[tri[:, 1]] + accel[tri[:, 2]]) / 3
                            ps = ps + self.probe * (am * n).sum(1)
                        f = f - ps[:, None] * n
                    load = load + f * on[:, None]
                T.append(load * area[:, None])
        cat = lambda q: torch.cat(q) if q else None
        U = cat(U)
        F = None
        if interp:
            F = ((v[self.tri[:, 0]] + v[self.tri[:, 1]] + v[self.tri[:, 2]]) / 3 - U) / self.dt
        return U, F, cat(T), cat(A), cat(tau)

    def spread(self, F, A, tau):
        n = self.n
        f = torch.zeros((3, n[0] * n[1] * n[2]), dtype=torch.float64, device=self.dev)
        cl = A * (sum(self.h) / 3) / (self.h[0] * self.h[1] * self.h[2])
        for o in range(0, len(A), CHUNK):
            q = slice(o, o + CHUNK)
            for i in range(3):
                at, phi = self.shape(tau[q], i)
                f[i].index_add_(0, at.reshape(-1), (phi * (cl[q] * F[q, i])[:, None]).reshape(-1))
        return [g.reshape(n[2], n[1], n[0]) for g in f]

    def accelerations(self, x, T, k, graph=False):
        ext = torch.zeros_like(x)
        for j in range(3):
            ext = ext.index_add(0, self.tri[:, j], T / 3)
        a = (ext + self.internal(x, k, graph)) / self.mass[self.owner][:, None]
        return torch.where(self.clamped[:, None], torch.zeros_like(a), a)

    def advance(self, x, v, T, k, graph=False):
        a = self.accelerations(x, T, k, graph)
        v1 = torch.where(self.clamped[:, None], torch.zeros_like(v), v + self.dt * a)
        return x + self.dt * v1, v1

    def state(self):
        i = self.i
        return tuple(None if t is None else t.double().T.contiguous() for t in (i.x, i.v, i.accel))

    def step(self, x, v, accel=None, spread=True):
        f = self.i.fields
        _, F, T, A, tau = self.markers(x, v, f, self.i.p, accel)
        x1, v1 = self.advance(x, v, T, self.k)
        return x1, v1, self.spread(F, A, tau) if spread else None

    # the fluid
    def eig(self):
        out = []
        for d, ax in enumerate((2, 1, 0)):
            k = torch.arange(self.n[d] // 2 + 1 if d == 0 else self.n[d], dtype=torch.float64,
                             device=self.dev)
            lam = -(4 / self.h[d] ** 2) * torch.sin(math.pi * k / self.n[d]) ** 2
            out.append(lam.reshape([-1 if q == ax else 1 for q in range(3)]))
        return out

    def flow_step(self, nu, forcing=None):
        h, dt = self.h, self.dt
        sh = lambda f, d, s: torch.roll(f, -s, dims=(2, 1, 0)[d])
        u = [f.double() for f in self.i.fields]
        p = self.i.p.double()
        lam = self.eig()
        lap = lambda f: sum((sh(f, d, 1) - 2 * f + sh(f, d, -1)) / h[d] ** 2 for d in range(3))
        Hp, force = None, None
        for l in range(3):
            al = GAMMA[l] + RHO[l]
            a = al * dt * nu / 2
            H, new = [], []
            for c in range(3):
                acc = 0.0
                for d in range(3):
                    if c == d:
                        q = (0.5 * (u[c] + sh(u[c], c, 1))) ** 2
                        acc = acc + (q - sh(q, c, -1)) / h[c]
                    else:
                        q = 0.25 * (u[d] + sh(u[d], c, -1)) * (u[c] + sh(u[c], d, -1))
                        acc = acc + (sh(q, d, 1) - q) / h[d]
                H.append(-acc)
            for c in range(3):
                r = GAMMA[l] * H[c] - al * (p - sh(p, c, -1)) / h[c] + al * nu * lap(u[c])
                if RHO[l]:
                    r = r + RHO[l] * Hp[c]
                R = torch.fft.rfftn(dt * r)
                for d in range(3):
                    R = R / (1 - a * lam[d])
                new.append(u[c] + torch.fft.irfftn(R, s=r.shape))
            Hp, u = H, new
            if forcing is not None:
                force = forcing(u)
                u = [q + dt * f for q, f in zip(u, force)]
            div = sum((sh(u[d], d, 1) - u[d]) / h[d] for d in range(3)) / (al * dt)
            tot = lam[0] + lam[1] + lam[2]
            tot[0, 0, 0] = 1.0
            P = torch.fft.rfftn(div) / tot
            P[0, 0, 0] = 0.0
            phi = torch.fft.irfftn(P, s=div.shape)
            u = [u[d] - al * dt * (phi - sh(phi, d, -1)) / h[d] for d in range(3)]
            p = p + phi - a * lap(phi)
        return u, p, force


def _edges(tri):
    """[E, 4] (a, b, c, d): the edge, the wing of the face holding a -> b and
    that of the face holding b -> a (a large negative number if there is none)."""
    t = np.asarray(tri, np.int64)
    half = np.concatenate([t[:, [0, 1, 2]], t[:, [1, 2, 0]], t[:, [2, 0, 1]]])
    m = int(t.max()) + 1
    fwd = half[:, 0] * m + half[:, 1]
    order = np.argsort(fwd)
    back = half[:, 1] * m + half[:, 0]
    at = np.minimum(np.searchsorted(fwd[order], back), len(fwd) - 1)
    found = fwd[order][at] == back
    other = np.where(found, half[order][at, 2], -(1 << 40))
    keep = (half[:, 0] < half[:, 1]) | ~found
    return np.concatenate([half, other[:, None]], 1)[keep]


def exact(case, seed):
    kind = case["kind"]
    e = Exact(case, seed)
    out = lambda t: t.T.contiguous()
    with torch.no_grad():
        if kind == "flow":
            u, p, _ = e.flow_step(case["nu"])
            return {"u": u, "p": p}
        x, v, accel = e.state()
        if kind in ("step", "host"):
            x1, v1, f = e.step(x, v, accel)
            return {"x": out(x1), "v": out(v1), "f": f}
        if kind == "graph":
            x, v, _ = e.step(x, v, spread=False)
            x1, v1, f = e.step(x, v)
            return {"x": out(x1), "v": out(v1), "f": f}
        if kind == "transfer":
            U, F, T, A, tau = e.markers(x, v, e.i.fields, e.i.p, accel)
            return {"U": out(U), "F_marker": out(F), "F_ext": out(T), "f": e.spread(F, A, tau)}
        if kind == "forces":
            return {"F": out(e.internal(x, e.k))}
        if kind == "pc":       # the first step after creation is a classical Runge-Kutta step
            _, F, T, A, tau = e.markers(x, v, e.i.fields)
            acc = lambda y: e.accelerations(y, e.markers(y, v, e.i.fields, interp=False)[2], e.k)
            h = e.dt
            a1 = e.accelerations(x, T, e.k)
            v2 = v + h / 2 * a1
            a2 = acc(x + h / 2 * v)
            v3 = v + h / 2 * a2
            a3 = acc(x + h / 2 * v2)
            v4 = v + h * a3
            a4 = acc(x + h * v3)
            return {"x": out(x + h / 6 * (v + 2 * v2 + 2 * v3 + v4)),
                    "v": out(v + h / 6 * (a1 + 2 * a2 + 2 * a3 + a4)), "f": e.spread(F, A, tau)}
        if kind == "coupled":
            def forcing(u):
                _, F, _, A, tau = e.markers(x, v, u, probe=False)
                return e.spread(F, A, tau)
            u, p, f = e.flow_step(case["nu"], forcing)
            T = e.markers(x, v, u, p, interp=False)[2]
            x1, v1 = e.advance(x, v, T, e.k)
            return {"u": u, "p": p, "x": out(x1), "v": out(v1), "f": f}
    # rollout: reverse mode through the steps, each recomputed
    k = e.i.k.double().to(e.dev)

    def one(x, v, k):
        T = e.markers(x, v, e.i.fields, interp=False)[2]
        return e.advance(x, v, T, k, graph=True)
    leaf = [t.detach().requires_grad_() for t in (x, v, k)]
    y = leaf[:2]
    states = []
    with torch.no_grad():
        for _ in range(case["steps"]):
            states.append(y)
            with torch.enable_grad():
                a, b = (t.detach().requires_grad_() for t in y)
                y = [t.detach() for t in one(a, b, k)]
    g = [c.double().T.contiguous() for c in e.i.cot]
    gk = torch.zeros_like(k)
    for a, b in reversed(states):
        a, b, kk = (t.detach().requires_grad_() for t in (a, b, k))
        ga, gb, q = torch.autograd.grad(one(a, b, kk), (a, b, kk), g)
        g, gk = [ga, gb], gk + q
    return {"x": out(y[0]), "v": out(y[1]), "gx": out(g[0]), "gv": out(g[1]), "gk": gk.cpu()}
