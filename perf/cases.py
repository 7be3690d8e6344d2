"""The work that users of the library have it do, as measurable cases.

Every case goes through the package's public entry points (Body, Batch, the
union of bodies and the energy's autograd function) on seeded particle sets
of this repository's own workloads: lattices and generated sets with a
jitter of +-0.25 dx, h = 1.3 dx.  A case is a dict of plain values:

  kind   "relax"     one body, its own launches (Body.relax)
         "graph"     a batch of bodies, iterations replayed from a CUDA graph
         "monitor"   Body.relax, then the uniformity statistics of the result
         "descent"   Body.relax_energy: the energy-descent relaxation
         "gradient"  the uniformity energy, its forward and its backward
         "generate"  Body.map_particles: the initial set of a body
  shape  the geometry; dx the particle spacing; iters the iterations a pass

A pass holds few iterations: a particle pressed against a wall is accepted or
sent back on the last bit, and over tens of iterations two correct roundings
part by a whole step there.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_2501_03056_gb300 as fppg
from paper_2501_03056_gb300 import autograd
from paper_2501_03056_gb300 import workloads as W

PAIRS = 72.6           # neighbours within 2h = 2.6 dx of a volume particle
FLOPS_PER_PAIR = 20    # difference, distance, root, weight, accumulation


def listed():
    return [
        # the smallest call: the unit cube's 10.6 k particles (all four moving
        # or fixed feature classes), where launches and latency count
        {"name": "cube 10k relax", "kind": "relax", "shape": "cube", "dx": 0.05, "iters": 10},
        # many tiny bodies at once: what the batched form is for
        {"name": "8 small bodies graph", "kind": "graph", "shape": "small", "bodies": 8, "dx": 0.06, "iters": 8},
        # two overlapping bodies united (partner rules, a shared grid)
        {"name": "union pair graph", "kind": "graph", "shape": "union", "dx": 0.03, "iters": 10},
        # the mid-size workload of the benchmark: icosphere and torus, 0.8 M
        {"name": "sphere+torus graph", "kind": "graph", "shape": "sphere_torus", "dx": 0.02, "iters": 4},
        # a thin mobile band under a mesh with features, generated, 2.4 M
        {"name": "gear graph", "kind": "graph", "shape": "gear", "dx": 0.004, "iters": 10},
        # the 64 uneven bodies of the benchmark with their unions, 7.1 M
        {"name": "64 bodies graph", "kind": "graph", "shape": "assemblies", "bodies": 64, "dx": 0.008, "iters": 4},
        # the headline: the vehicle shell filled with 19 M particles
        {"name": "vehicle graph", "kind": "graph", "shape": "vehicle", "dx": 0.0068, "iters": 5},
        # relaxing in chunks and watching the uniformity statistics
        {"name": "sphere monitor", "kind": "monitor", "shape": "sphere", "dx": 0.02, "iters": 4},
        # the energy and its gradients by position and mesh vertex (a
        # differentiable loss term), as the benchmark's backward leg
        {"name": "torus gradient", "kind": "gradient", "shape": "torus", "dx": 0.02, "iters": 1},
        # the energy-descent relaxation beside the paper's force
        {"name": "sphere descent", "kind": "descent", "shape": "sphere", "dx": 0.02, "iters": 5},
        # the initial set of a body from its mesh: features, surface, volume
        {"name": "gear generate", "kind": "generate", "shape": "gear", "dx": 0.004, "iters": 1},
    ]


# per kind: the shapes it is used on and, per shape, the range of dx
RANGES = {
    "relax": {"cube": (0.012, 0.1), "sphere": (0.015, 0.12), "torus": (0.011, 0.1)},
    "graph": {"cube": (0.012, 0.1), "small": (0.04, 0.09), "union": (0.012, 0.06), "sphere": (0.009, 0.06),
              "sphere_torus": (0.012, 0.08), "gear": (0.0032, 0.02), "assemblies": (0.009, 0.02),
              "vehicle": (0.0075, 0.025)},
    "monitor": {"cube": (0.012, 0.1), "sphere": (0.012, 0.08), "torus": (0.01, 0.08)},
    "gradient": {"cube": (0.015, 0.1), "sphere": (0.015, 0.1), "torus": (0.011, 0.08)},
    "descent": {"cube": (0.015, 0.1), "sphere": (0.015, 0.1), "torus": (0.011, 0.08)},
    "generate": {"gear": (0.0035, 0.02), "vehicle": (0.01, 0.03), "sphere": (0.008, 0.05)},
}
KINDS = ("relax", "graph", "graph", "graph", "graph", "monitor", "gradient", "descent", "generate")


def draw(rng):
    kind = rng.choice(KINDS)
    shape = rng.choice(sorted(RANGES[kind]))
    lo, hi = RANGES[kind][shape]
    c = {"kind": kind, "shape": shape, "dx": round(math.exp(rng.uniform(math.log(lo), math.log(hi))), 6),
         "iters": 1 if kind in ("gradient", "generate") else rng.randint(2, 5)}
    if shape == "small":
        c["bodies"] = rng.randint(2, 24)
    if shape == "assemblies":
        c["bodies"] = rng.randint(5, 60)
    return c


# ---- inputs ------------------------------------------------------------------
SMALL = ("cube", "sphere", "torus")
BAND = {"band_cells": 2, "inner_cells": 1}    # the gear's relaxing and fixed layers


@functools.lru_cache(maxsize=None)
def mesh(shape):
    """(vertices, triangles, feature threshold in degrees) of a shape"""
    if shape == "cube":
        return (*W.cube_mesh(), 30.0)
    if shape == "sphere":
        return (*W.icosphere_mesh(5), None)
    if shape == "torus":
        return (*W.torus_mesh(1.0, 0.3, 256, 64), None)
    if shape == "gear":
        return (*W.gear_mesh(), 30.0)
    if shape == "vehicle":    # 0.5 M triangles with their seeded noise
        return (*W.vehicle_mesh(spacing=0.042), 30.0)
    raise ValueError(shape)


def _uniform(gen, n, m, amp):
    return (torch.rand((n, m), generator=gen, device="cuda", dtype=torch.float64) * 2 - 1) * amp


def _lattice(lo, hi, dx, shift):
    ax = [torch.arange(math.floor(lo[k] / dx), math.ceil(hi[k] / dx) + 1, device="cuda", dtype=torch.float64) * dx
          + shift * dx for k in range(3)]
    return torch.stack([g.reshape(-1) for g in torch.meshgrid(*ax, indexing="ij")], 1)


def _cube_particles(dx, gen):
    n = int(round(1.0 / dx))
    d = 1.0 / n
    k = (torch.arange(n, device="cuda", dtype=torch.float64) + 0.5) * d - 0.5
    a, b = (g.reshape(-1) for g in torch.meshgrid(k, k, indexing="ij"))
    e = torch.arange(1, n, device="cuda", dtype=torch.float64) * d - 0.5
    xyz, cls = [], []
    for axis in range(3):
        o1, o2 = [ax for ax in range(3) if ax != axis]
        for sg in (-0.5, 0.5):
            p = torch.empty((n * n, 3), device="cuda", dtype=torch.float64)
            j = _uniform(gen, n * n, 2, 0.25 * d)
            p[:, axis], p[:, o1], p[:, o2] = sg, a + j[:, 0], b + j[:, 1]
            xyz.append(p)
            cls.append(fppg.S)
    for axis in range(3):
        o1, o2 = [ax for ax in range(3) if ax != axis]
        for s1 in (-0.5, 0.5):
            for s2 in (-0.5, 0.5):
                p = torch.empty((n - 1, 3), device="cuda", dtype=torch.float64)
                p[:, axis], p[:, o1], p[:, o2] = e + _uniform(gen, n - 1, 1, 0.25 * d)[:, 0], s1, s2
                xyz.append(p)
                cls.append(fppg.F)
    xyz.append(torch.tensor([[x, y, z] for x in (-0.5, 0.5) for y in (-0.5, 0.5) for z in (-0.5, 0.5)],
                            device="cuda", dtype=torch.float64))
    cls.append(fppg.P)
    g = torch.stack([t.reshape(-1) for t in torch.meshgrid(k, k, k, indexing="ij")], 1)
    xyz.append(g + _uniform(gen, len(g), 3, 0.25 * d))
    cls.append(fppg.V)
    return xyz, cls


def _sphere_particles(dx, gen, r):
    ns = int(round(4 * math.pi * r * r / (dx * dx)))
    k = torch.arange(ns, device="cuda", dtype=torch.float64)
    z = 1 - (2 * k + 1) / ns
    rho, phi = torch.sqrt(1 - z * z), k * (math.pi * (3 - math.sqrt(5)))
    s = torch.stack([rho * torch.cos(phi), rho * torch.sin(phi), z], 1) * r + _uniform(gen, ns, 3, 0.25 * dx)
    s = s * (r / s.norm(dim=1, keepdim=True))
    v = _lattice((-r,) * 3, (r,) * 3, dx, 0.0)
    v = v[v.norm(dim=1) <= r - 0.5 * dx]
    return [s, v + _uniform(gen, len(v), 3, 0.25 * dx)], [fppg.S, fppg.V]


def _torus_particles(dx, gen, R=1.0, r=0.3):
    pts = []
    nv = int(round(2 * math.pi * r / dx))
    for j in range(nv):
        v = 2 * math.pi * (j + 0.5) / nv
        nu = int(round(2 * math.pi * (R + r * math.cos(v)) / dx))
        u = 2 * math.pi * (torch.arange(nu, device="cuda", dtype=torch.float64) + 0.5 * (j % 2)) / nu
        pts.append(torch.stack([u, torch.full_like(u, v)], 1))
    uv = torch.cat(pts)
    uv = uv + _uniform(gen, len(uv), 2, 0.25 * dx) / torch.tensor([R, r], device="cuda", dtype=torch.float64)
    rho = R + r * torch.cos(uv[:, 1])
    s = torch.stack([rho * torch.cos(uv[:, 0]), rho * torch.sin(uv[:, 0]), r * torch.sin(uv[:, 1])], 1)
    v = _lattice((-R - r, -R - r, -r), (R + r, R + r, r), dx, 0.0)
    tube = ((v[:, :2].norm(dim=1) - R) ** 2 + v[:, 2] ** 2).sqrt()
    v = v[tube <= r - 0.5 * dx]
    return [s, v + _uniform(gen, len(v), 3, 0.25 * dx)], [fppg.S, fppg.V]


def particles(shape, dx, seed, radius=1.0):
    """(xyz float32 [n, 3], class int32 [n]) of a lattice-filled shape, on the host"""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    xyz, cls = (_cube_particles(dx, gen) if shape == "cube" else
                _sphere_particles(dx, gen, radius) if shape == "sphere" else _torus_particles(dx, gen))
    c = np.concatenate([np.full(len(x), k, np.int32) for x, k in zip(xyz, cls)])
    return torch.cat(xyz).float().cpu().numpy(), c


def spacing(dx):
    """(dx, h = 1.3 dx) as FP32 values"""
    return float(np.float32(dx)), W.smoothing_length(dx)


def _body(verts, tris, dihedral, dx, stream):
    b = fppg.Body(verts, tris, *spacing(dx), stream=stream)
    if dihedral is not None:
        b.extract_features(dihedral)
    return b


def filled(shape, dx, seed, stream):
    """A body with its lattice particles"""
    v, t, deg = mesh(shape)
    b = _body(v, t, deg, dx, stream)
    b.set_particles(*particles(shape, dx, seed))
    return b


def jitter(b, dx, seed):
    """The relaxing volume particles of a generated body moved by +-0.25 dx
    (they stay inside their cells)"""
    xyz, cls, cons = b.get_particles()
    gen = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.from_numpy(xyz).cuda()
    j = torch.rand(x.shape, generator=gen, device="cuda") - 0.5
    x += j * (0.5 * float(np.float32(dx))) * (torch.from_numpy(cls).cuda() == fppg.V)[:, None]
    b.set_particles(x.cpu().numpy(), cls)
    b.set_constraints(cons)


def generated(v, t, deg, dx, stream, **options):
    """A body with the particles of its own generation"""
    b = _body(v, t, deg, dx, stream)
    b.map_particles(**options)
    return b


def _bodies(case, seed, stream):
    """The bodies of a relaxation case"""
    shape, dx = case["shape"], case["dx"]
    if shape in SMALL:
        return [filled(shape, dx, seed, stream)]
    if shape == "sphere_torus":
        return [filled("sphere", dx, seed, stream), filled("torus", dx, seed + 1000003, stream)]
    if shape == "small":
        return [filled(SMALL[k % 3], dx * (1.0 + 0.07 * (k % 5)), seed + 1000003 * k, stream)
                for k in range(case["bodies"])]
    if shape in ("gear", "vehicle"):
        b = generated(*mesh(shape), dx, stream, **(BAND if shape == "gear" else {}))
        jitter(b, dx, seed)
        return [b]
    if shape == "union":
        cv, ct, deg = mesh("cube")
        a = _body(cv, ct, deg, dx, stream)
        a.map_particles()
        sv, st = W.icosphere_mesh(3, 0.35)
        b = _body((sv + np.array([0.45, 0.05, -0.03])).astype(np.float32), st, None, dx, stream)
        b.map_particles()
        fppg.union(a, b)
        jitter(a, dx, seed)
        jitter(b, dx, seed + 1000003)
        return [a, b]
    if shape == "assemblies":
        asm = W.batch_union_workload(bodies=case["bodies"], dx=dx)
        out = [generated(a.verts, a.tris, a.dihedral_deg, dx, stream, **a.meta["generate"]) for a in asm]
        for k, a in enumerate(asm):
            if a.meta.get("union_with", -1) > k:
                fppg.union(out[k], out[a.meta["union_with"]])
        for k, b in enumerate(out):
            jitter(b, dx, seed + 1000003 * k)
        return out
    raise ValueError(shape)


def _torus_triangles(xyz, cls):
    """The mesh triangle under each surface particle of the torus (-1 for the
    others), from its angles: what a user who placed them there knows"""
    u = np.mod(np.arctan2(xyz[:, 1], xyz[:, 0]), 2 * np.pi) * (256 / (2 * np.pi))
    w = np.mod(np.arctan2(xyz[:, 2], np.hypot(xyz[:, 0], xyz[:, 1]) - 1.0), 2 * np.pi) * (64 / (2 * np.pi))
    i, j = np.minimum(u.astype(np.int64), 255), np.minimum(w.astype(np.int64), 63)
    t = 2 * (i * 64 + j) + (w - j > u - i)
    return np.where(cls == fppg.S, t, -1).astype(np.int32)


def _nearest_triangles(shape, xyz, cls):
    """The constraint triangles of a gradient case's surface particles"""
    if shape == "torus":
        return _torus_triangles(xyz, cls)
    v, t, _ = mesh(shape)
    tri = torch.from_numpy(v.astype(np.float64)).cuda()[torch.from_numpy(t.astype(np.int64)).cuda()]
    out = np.full(len(xyz), -1, np.int32)
    s = np.flatnonzero(cls == fppg.S)
    x = torch.from_numpy(xyz[s].astype(np.float64)).cuda()
    got = [_surface_choice(x[k:k + 2048], tri, float("inf"), 1e-6)[0] for k in range(0, len(s), 2048)]
    out[s] = torch.cat(got).cpu().numpy() if got else 0
    return out


def prepare(case, seed):
    stream = torch.cuda.current_stream()
    kind, shape, dx = case["kind"], case["shape"], case["dx"]
    state = {"case": case}
    if kind == "generate":
        # a mesh of its own for each seed: the shape turned about z and y
        rng = np.random.default_rng(seed)
        v, t, deg = mesh(shape)
        a, b = rng.uniform(0, 2 * np.pi, 2)
        rz = np.array([[np.cos(a), -np.sin(a), 0], [np.sin(a), np.cos(a), 0], [0, 0, 1]])
        ry = np.array([[np.cos(b), 0, np.sin(b)], [0, 1, 0], [-np.sin(b), 0, np.cos(b)]])
        state["body"] = _body((v @ (ry @ rz).T).astype(np.float32), t, deg, dx, stream)
        # room for any turn's count, the rows after it left at zero
        state["out"] = torch.zeros((int(2.5 * _count(shape, dx, 1)[2]), 3), device="cuda")
    elif kind == "gradient":
        v, t, deg = mesh(shape)
        b = _body(v, t, deg, dx, stream)
        xyz, cls = particles(shape, dx, seed)
        b.set_particles(xyz, cls)
        b.set_constraints(_nearest_triangles(shape, xyz, cls))
        state["body"] = b
        state["y"] = torch.from_numpy(xyz).cuda().requires_grad_(True)
        state["verts"] = torch.from_numpy(v).cuda().requires_grad_(True)
    elif kind == "graph":
        bodies = _bodies(case, seed, stream)
        state["bodies"] = bodies
        state["batch"] = fppg.Batch(bodies, stream=stream)
        state["batch"].set_graph_iters(case["iters"])
        state["out"] = [torch.empty((b.n, 3), device="cuda") for b in bodies]
    else:
        state["body"] = filled(shape, dx, seed, stream)
        state["out"] = torch.empty((state["body"].n, 3), device="cuda")
    return state


def run(state):
    case = state["case"]
    kind, iters = case["kind"], case["iters"]
    if kind == "graph":
        state["batch"].relax(iters, use_graph=True)
        state["batch"].store()
        for b, o in zip(state["bodies"], state["out"]):
            b.copy_positions_dev(o.data_ptr())
        return state["out"]
    body = state["body"]
    if kind == "generate":
        n = body.map_particles(**(BAND if case["shape"] == "gear" else {}))
        if n <= len(state["out"]):
            body.copy_positions_dev(state["out"].data_ptr())
        return {"n": n, "xyz": state["out"]}
    if kind == "gradient":
        y, verts = state["y"], state["verts"]
        e = autograd.uniformity_energy(y, verts, body)
        gy, gv = torch.autograd.grad(e, (y, verts))
        # the densities under the sum are FP32
        return {"energy": e.detach().float(), "dy": gy, "dverts": gv}
    if kind == "descent":
        body.relax_energy(iters)
    else:
        body.relax(iters)
    body.copy_positions_dev(state["out"].data_ptr())
    if kind == "monitor":
        return {"xyz": state["out"], "stats": body.stats()}
    return state["out"]


# ---- what a pass cannot do without ----------------------------------------------
def _count(shape, dx, bodies):
    """(surface, relaxing volume, all) particles of a shape, about"""
    area, vol = {"cube": (6.0, 1.0), "sphere": (12.57, 4.19), "torus": (11.84, 1.78), "gear": (7.0, 0.72),
                 "vehicle": (21.6, 5.68), "union": (6.6, 1.11)}.get(shape, (0.0, 0.0))
    if shape == "sphere_torus":
        area, vol = 24.4, 5.97
    elif shape == "small":
        area, vol = 10.1 * bodies / 1.3, 2.3 * bodies / 1.5
    elif shape == "assemblies":
        area, vol = 1.4 * bodies, 0.055 * bodies
    s, v = area / dx ** 2, vol / dx ** 3
    if shape in ("gear", "assemblies"):      # only a band under the surface relaxes
        band = 2 if shape == "gear" else 3
        return s, min(v, s * band), s + min(v, s * (band + 1))
    return s, v, s + v


def work(case):
    s, v, n = _count(case["shape"], case["dx"], case.get("bodies", 1))
    if case["kind"] == "generate":
        return {"bytes": 16.0 * n + 36.0 * len(mesh(case["shape"])[1]), "flops": 10.0 * n}
    pairs = v * PAIRS + s * 20.2
    if case["kind"] == "gradient":
        nv = len(mesh(case["shape"])[0])
        return {"bytes": 28.0 * n + 24.0 * nv, "flops": 2 * pairs * FLOPS_PER_PAIR}
    per = 2 * FLOPS_PER_PAIR if case["kind"] == "descent" else FLOPS_PER_PAIR
    # positions, classes and constraints in, positions and constraints out
    f = case["iters"] * pairs * per + (pairs * FLOPS_PER_PAIR if case["kind"] == "monitor" else 0)
    return {"bytes": 36.0 * n, "flops": f}


# ---- the same in 64 bits -----------------------------------------------------------
# Plain torch on the method's formulas, for the bodies with analytic shapes:
# neighbours by cells, triangles by brute force.
ACTS = torch.tensor([[1, 0, 1, 0, 1], [1, 1, 1, 1, 1], [0, 0, 1, 0, 1], [0, 0, 0, 0, 0], [0, 0, 0, 0, 0]],
                    dtype=torch.bool)    # ACTS[i, j]: class j acts on class i


def _pairs(x, cls, reach):
    """Blocks of (i, j, q = x_j - x_i, r) with r < reach, j acting on i, i != j"""
    acts = ACTS.to(x.device)
    lo = x.amin(0)
    c = ((x - lo) / reach).long() + 1
    n = c.amax(0) + 2
    key = (c[:, 2] * n[1] + c[:, 1]) * n[0] + c[:, 0]
    order = torch.argsort(key)
    skey = key[order]
    block = 200000
    for a in range(0, len(x), block):
        i0 = order[a:a + block]
        for dz in (-1, 0, 1):
            for dy in (-1, 0, 1):
                k = key[i0] + (dz * n[1] + dy) * n[0]
                s, e = torch.searchsorted(skey, k - 1), torch.searchsorted(skey, k + 2)
                m = e - s
                i = torch.repeat_interleave(i0, m)
                off = torch.arange(int(m.sum()), device=x.device) - torch.repeat_interleave(m.cumsum(0) - m, m)
                j = order[torch.repeat_interleave(s, m) + off]
                q = x[j] - x[i]
                r = q.norm(dim=1)
                w = (r < reach) & (i != j) & acts[cls[i], cls[j]]
                yield i[w], j[w], q[w], r[w]


def _alpha(h):
    return 21.0 / (16.0 * math.pi * h ** 3)


def _density(x, cls, h):
    rho = torch.full((len(x),), _alpha(h), dtype=torch.float64, device=x.device)
    rmin = float("inf")
    for i, j, q, r in _pairs(x, cls, 2 * h):
        t = 1 - r / (2 * h)
        rho.index_add_(0, i, _alpha(h) * t ** 4 * (2 * r / h + 1))
        k = cls[i] <= 2
        if bool(k.any()):
            rmin = min(rmin, float(r[k].min()))
    return rho, rmin


def _lattice_sum(dx, h, dim):
    m = int(math.ceil(2 * h / dx)) + 1
    k = range(-m, m + 1)
    tot = 0.0
    for a in k:
        for b in (k if dim > 1 else (0,)):
            for c in (k if dim > 2 else (0,)):
                r = dx * math.sqrt(a * a + b * b + c * c)
                tot += _alpha(h) * max(1 - r / (2 * h), 0.0) ** 4 * (2 * r / h + 1)
    return tot


def _ideal(cls, dx, h):
    w0 = torch.tensor([_lattice_sum(dx, h, 2), _lattice_sum(dx, h, 3), _lattice_sum(dx, h, 1), 0.0, 0.0],
                      dtype=torch.float64, device=cls.device)
    return w0[cls]


def _repulsion(x, cls, h):
    """Eq. 15 up to its constant (the step divides it out)"""
    a = torch.zeros_like(x)
    for i, j, q, r in _pairs(x, cls, 2 * h):
        a.index_add_(0, i, -((1 - r / (2 * h)) ** 3)[:, None] * q)
    return a


def _energy_gradient(x, cls, dx, h):
    """dE/dx of E = sum over moving particles of (rho - W0)^2, and E"""
    rho, _ = _density(x, cls, h)
    d = torch.where(cls <= 2, rho - _ideal(cls, dx, h), 0.0)
    g = torch.zeros_like(x)
    for i, j, q, r in _pairs(x, cls, 2 * h):
        # dW/dr = -(5 alpha / h^2) r (1 - r / 2h)^3
        f = (2 * d[i] * 5 * _alpha(h) / (h * h) * (1 - r / (2 * h)) ** 3)[:, None] * q
        g.index_add_(0, i, f)
        g.index_add_(0, j, -f)
    return g, (d * d).sum()


def _surface_choice(y, tri, limit, tol):
    """(triangle, foot) of the closest triangle, by plane distance within
    limit, whose foot lies inside it; -1 for none"""
    a, b, c = tri[:, 0], tri[:, 1], tri[:, 2]
    n = torch.linalg.cross(b - a, c - a)
    n = n / n.norm(dim=1, keepdim=True)
    ok = torch.ones((len(y), len(tri)), dtype=torch.bool, device=y.device)
    for p, q in ((a, b), (b, c), (c, a)):
        m = torch.linalg.cross(n, q - p)
        m = m / m.norm(dim=1, keepdim=True)
        ok &= y @ m.T - (p * m).sum(1) >= -tol
    d = y @ n.T - (a * n).sum(1)
    ok &= d.abs() <= limit
    best = torch.where(ok, d.abs(), torch.inf)
    t = best.argmin(1)
    found = ok.any(1)
    k = torch.arange(len(y), device=y.device)
    return torch.where(found, t, -1), y - torch.where(found, d[k, t], 0.0)[:, None] * n[t]


def _outside(y, tri):
    """Whether y lies outside: sign by the pseudonormal of the closest feature"""
    a, b, c = tri[:, 0], tri[:, 1], tri[:, 2]
    ab, ac = b - a, c - a
    nrm = torch.linalg.cross(ab, ac)
    nrm = nrm / nrm.norm(dim=1, keepdim=True)

    def to_edge(p, q):
        e = q - p
        t = ((y @ e.T - (p * e).sum(1)) / (e * e).sum(1)).clamp(0, 1)
        return ((y[:, None] - p) - t[..., None] * e).square().sum(-1)

    d = y @ nrm.T - (a * nrm).sum(1)
    inside = torch.ones_like(d, dtype=torch.bool)
    for p, q in ((a, b), (b, c), (c, a)):
        m = torch.linalg.cross(nrm, q - p)
        inside &= y @ m.T - (p * m).sum(1) >= 0
    best = torch.where(inside, d * d, torch.inf)
    for p, q in ((a, b), (b, c), (c, a)):
        best = torch.minimum(best, to_edge(p, q))
    near = best.amin(1)
    # the pseudonormal of the closest feature points as the sum of the normals
    # of the triangles that touch it, by their angle there
    touch = best <= (near * (1 + 1e-9) + 1e-24)[:, None]
    k = torch.arange(len(y), device=y.device)
    t = best.argmin(1)
    foot = torch.where(inside[k, t][:, None], y - d[k, t][:, None] * nrm[t], 0.0)
    for p, q in ((a, b), (b, c), (c, a)):
        e = q[t] - p[t]
        u = (((y - p[t]) * e).sum(1) / (e * e).sum(1)).clamp(0, 1)
        f = p[t] + u[:, None] * e
        take = ~inside[k, t] & ((y - f).square().sum(1) <= best[k, t] * (1 + 1e-9) + 1e-24)
        foot = torch.where(take[:, None], f, foot)
    w = torch.zeros_like(best)
    for p, q, r in ((a, b, c), (b, c, a), (c, a, b)):
        at = (foot[:, None] - p).square().sum(-1) < 1e-20
        cosang = ((q - p) * (r - p)).sum(1) / ((q - p).norm(dim=1) * (r - p).norm(dim=1))
        w = torch.where(at, torch.arccos(cosang)[None], w)
    w = torch.where((w == 0) & touch, 1.0, w) * touch
    psi = w @ nrm
    return ((y - foot) * psi).sum(1) > 0


def _near_surface(shape, x, dx):
    if shape == "cube":
        return x.abs().amax(1) > 0.5 - 2 * dx
    if shape == "sphere":
        return x.norm(dim=1) > 1.0 - 2 * dx
    return ((x[:, :2].norm(dim=1) - 1.0) ** 2 + x[:, 2] ** 2).sqrt() > 0.3 - 2 * dx


def _relaxed(shape, dx, seed, iters, descent):
    """(positions, classes, largest last move) after iters iterations"""
    xyz, c = particles(shape, dx, seed)
    d, h = spacing(dx)
    x = torch.from_numpy(xyz.astype(np.float64)).cuda()
    cls = torch.from_numpy(c.astype(np.int64)).cuda()
    v, t, _ = mesh(shape)
    v64 = torch.from_numpy(v.astype(np.float64)).cuda()
    faces = torch.from_numpy(t.astype(np.int64)).cuda()
    tri = v64[faces]
    tol = 2.0 ** -20 * float((v64.amax(0) - v64.amin(0)).max())
    a, b, e = tri[:, 0], tri[:, 1], tri[:, 2]
    nrm = torch.linalg.cross(b - a, e - a)
    nrm = nrm / nrm.norm(dim=1, keepdim=True)
    S, V, F = (torch.nonzero(cls == k)[:, 0] for k in (0, 1, 2))
    cons = torch.full((len(x),), -1, dtype=torch.long, device=x.device)
    # a feature particle of the cube slides along its edge: the free axis
    free = (x[F].abs() < 0.5).double()
    move = torch.zeros(len(x), dtype=torch.float64, device=x.device)
    per = max(1, 20_000_000 // len(tri))
    for _ in range(iters):
        acc = -_energy_gradient(x, cls, d, h)[0] if descent else _repulsion(x, cls, h)
        acc[cls > 2] = 0
        amax = float(acc.norm(dim=1).max())
        step = acc * ((h / 16) / amax if amax > 0 else 0.0)
        held = cons[S] >= 0
        n = nrm[cons[S].clamp(min=0)]
        sd = step[S]
        step[S] = torch.where(held[:, None], sd - (sd * n).sum(1, keepdim=True) * n, sd)
        y = x + step
        new = x.clone()
        for k in range(0, len(S), per):
            i = S[k:k + per]
            got, foot = _surface_choice(y[i], tri, 2 * d, tol)
            new[i] = torch.where((got >= 0)[:, None], foot, x[i])
            cons[i] = torch.where(got >= 0, got, cons[i])
        ok = torch.ones(len(V), dtype=torch.bool, device=x.device)
        near = torch.nonzero(_near_surface(shape, y[V], d))[:, 0]
        for k in range(0, len(near), per // 4 + 1):
            i = near[k:k + per // 4 + 1]
            ok[i] = ~_outside(y[V[i]], tri)
        new[V] = torch.where(ok[:, None], y[V], x[V])
        if len(F):
            new[F] = torch.where(free > 0, y[F].clamp(-0.5, 0.5), x[F])
        move = (new - x).norm(dim=1)
        x = new
    return x, cls, float(move.max())


def _statistics(x, cls, last, dx, h):
    rho, rmin = _density(x, cls, h)
    out = {}
    for k, name in ((0, "S"), (1, "V"), (2, "F")):
        r = rho[cls == k]
        out["n_" + name] = int(len(r))
        out["mean_" + name] = float(r.mean()) if len(r) else 0.0
        out["std_" + name] = float((r - r.mean()).square().mean().sqrt()) if len(r) else 0.0
    out["min_pair_over_dx"] = rmin / dx
    out["max_disp_over_dx"] = last / dx
    return out


def exact(case, seed):
    kind, shape, dx = case["kind"], case["shape"], case["dx"]
    _, v, n = _count(shape, dx, case.get("bodies", 1))
    d, h = spacing(dx)
    if kind == "gradient":
        xyz, c = particles(shape, dx, seed)
        cons = torch.from_numpy(_nearest_triangles(shape, xyz, c).astype(np.int64)).cuda()
        cls = torch.from_numpy(c.astype(np.int64)).cuda()
        mv, mt, _ = mesh(shape)
        y = torch.from_numpy(xyz.astype(np.float64)).cuda().requires_grad_(True)
        verts = torch.from_numpy(mv.astype(np.float64)).cuda().requires_grad_(True)
        tri = verts[torch.from_numpy(mt.astype(np.int64)).cuda()[cons.clamp(min=0)]]
        nrm = torch.linalg.cross(tri[:, 1] - tri[:, 0], tri[:, 2] - tri[:, 0])
        nrm = nrm / nrm.norm(dim=1, keepdim=True)
        x = y - torch.where(cons >= 0, ((y - tri[:, 0]) * nrm).sum(1), 0.0)[:, None] * nrm
        g, e = _energy_gradient(x.detach(), cls, d, h)
        gy, gv = torch.autograd.grad(x, (y, verts), g)
        return {"energy": e, "dy": gy, "dverts": gv}
    if kind == "graph" and shape in SMALL + ("sphere_torus",):
        parts = [("sphere", seed), ("torus", seed + 1000003)] if shape == "sphere_torus" else [(shape, seed)]
    elif kind in ("relax", "monitor", "descent"):
        parts = [(shape, seed)]
    else:
        return None     # the whole method: generation, features, Boolean partners
    # the brute-force surface tests and the pairs of the 64-bit units
    if case["iters"] * sum(1e-7 * _count(s, dx, 1)[1] * (3 if kind == "descent" else 1) +
                           8e-10 * _count(s, dx, 1)[0] * len(mesh(s)[1]) for s, _ in parts) > 8.5:
        return None
    if kind == "graph":
        return [_relaxed(s, dx, q, case["iters"], False)[0] for s, q in parts]
    x, cls, last = _relaxed(shape, dx, seed, case["iters"], kind == "descent")
    if kind == "monitor":
        return {"xyz": x, "stats": _statistics(x, cls, last, d, h)}
    return x
