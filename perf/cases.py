"""The work that programs have this library do, as cases that can be timed and compared.

A case is one call (or one short host loop) of the public Python binding on seeded synthetic
input of the kinds the repository's workloads use: spheres (smooth and rough), tori, periodic
height fields and open planes, with uniformly placed particles.  ``prepare`` builds what a
program holds before the call (mesh on the device, particle set, output buffers), ``run`` makes
the call, and ``exact`` gives the same result in plain 64-bit torch: straight rays unfolded
from every particle and every saddle vertex, then shortest chains of them.

The FP32 form carries single-precision distances and tangents in its double buffers; a program
that chooses it keeps single precision, so the real results of FP32 cases are float32.
Launch shapes are the library's own defaults: most programs never set or tune one.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_2404_19751_gb300 as css

DEV = "cuda"
POTENTIALS = {"harmonic": css.POT_HARMONIC, "wca": css.POT_WCA, "gaussian": css.POT_GAUSSIAN}
DYNAMICS = {"nve": css.INT_NVE, "bd": css.INT_BD, "abp": css.INT_ABP, "gd": css.INT_GD, "fire": css.INT_FIRE}


def _case(name, call, surface, size, particles, reach, precision="fp64", **more):
    """reach: the cutoff in world units, 0 for none.  size: sphere level, torus faces, or the
    grid points along one side."""
    c = dict(call=call, surface=surface, size=size, particles=particles, reach=reach, precision=precision,
             scale=1.0, noise=0.0, aspect=3.0, potential="harmonic", dynamics="none", steps=1, sets=1)
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: forces of a few dozen particles on a small rough sphere (latency, launches)
        _case("forces_ico3_n96_fp64", "forces", "sphere", 3, 96, 0.4, noise=0.01),
        # neighbour lists of a medium smooth sphere read back to the host for analysis
        _case("neighbors_ico5_n1024_fp64", "neighbors", "sphere", 5, 1024, 0.15),
        # a molecular-dynamics loop: constant-energy steps replayed as a graph, state read back
        _case("nve_ico5_n1024_fp32", "step", "sphere", 5, 1024, 0.15, "fp32", dynamics="nve", steps=10),
        # few sources, every pair, an open flat sheet: one source's whole mesh at a time
        _case("neighbors_plane21_n64_fp64", "neighbors", "plane", 21, 64, 0.0),
        # an odd number of particles on a torus, cutoff a few edges (the paper's N sweep)
        _case("neighbors_torus4592_n999_fp64", "neighbors", "torus", 4592, 999, 1.0),
        # every pair of 100 particles over a whole torus (the paper's V sweep, full mesh)
        _case("neighbors_torus4004_n100_fp64", "neighbors", "torus", 4004, 100, 0.0),
        # Brownian step on a fine periodic surface: the cutoff spans many faces
        _case("bd_hfield256_n8192_fp64", "step", "heightfield", 256, 8192, 0.05, dynamics="bd", potential="wca"),
        # many independent simulations advanced together
        _case("nve_tori16_batch_fp32", "batch", "torus", 0, 0, 0.1, "fp32", dynamics="nve", steps=2, sets=16),
        # one step of a large active simulation (soft discs), single-precision form
        _case("abp_noisy8_n65536_fp32", "step", "sphere", 8, 65536, 0.2244924, "fp32", scale=10.0, noise=0.02,
              dynamics="abp"),
        # forces of the same large rough sphere in double precision, hard potential
        _case("forces_noisy8_n65536_fp64", "forces", "sphere", 8, 65536, 0.2244924, scale=10.0, noise=0.02,
              potential="wca"),
        # the approximate solver: all pairs over a whole mesh
        _case("vhm_torus7992_n100", "vhm", "torus", 7992, 100, 0.0),
        # shortest paths as polylines, for the neighbours of about 40 particles
        _case("paths_noisy5_n2048", "paths", "sphere", 5, 2048, 0.15, noise=0.016),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """Sizes spread over the same ranges; the cutoff is drawn in mean edge lengths."""
    call = rng.choice(["forces", "forces", "neighbors", "neighbors", "step", "step", "batch", "vhm", "paths"])
    prec = "fp32" if call in ("forces", "step", "batch") and rng.random() < 0.5 else "fp64"
    if call == "batch":
        return _case("", "batch", "torus", 0, 0, _log(rng, 0.06, 0.15), prec, dynamics="nve", steps=rng.randint(1, 3),
                     sets=rng.randint(2, 16))
    if call == "vhm":
        return _case("", "vhm", "torus", int(_log(rng, 900, 8000)), int(_log(rng, 20, 100)), 0.0,
                     aspect=rng.uniform(2.0, 4.0))
    if call == "paths":
        return _case("", "paths", "sphere", rng.randint(3, 5), int(_log(rng, 300, 3000)), _log(rng, 0.1, 0.2),
                     noise=rng.uniform(0.005, 0.02))
    if call == "neighbors" and rng.random() < 0.3:   # every pair over a small mesh
        if rng.random() < 0.5:
            return _case("", "neighbors", "plane", rng.randint(9, 25), int(_log(rng, 17, 100)), 0.0)
        return _case("", "neighbors", "torus", int(_log(rng, 500, 4000)), int(_log(rng, 17, 100)), 0.0)
    surface = rng.choice(["sphere", "sphere", "torus", "heightfield", "plane"])
    edges = _log(rng, 2.5, 12.0)
    more = dict(potential="harmonic" if prec == "fp32" else rng.choice(["harmonic", "wca", "gaussian"]))
    if surface == "sphere":
        size = rng.randint(3, 7)
        scale = _log(rng, 1.0, 10.0)
        edge = 1.15 * scale / 2 ** size
        more.update(scale=scale, noise=rng.choice([0.0, rng.uniform(0.05, 0.4)]) * edge)
        faces = 20 * 4 ** size
    elif surface == "torus":
        faces = size = int(_log(rng, 1000, 60000))
        more.update(aspect=rng.uniform(2.0, 4.0))
        edge = math.sqrt(2 * 4 * math.pi ** 2 * more["aspect"] / faces)
    elif surface == "heightfield":
        size = rng.randint(32, 256)
        edge, faces = 1.2 / size, 2 * size * size
    else:
        size = rng.randint(9, 80)
        edge, faces = 1.0 / (size - 1), 2 * (size - 1) ** 2
    # no more unfoldings (particles x faces in reach) than the largest listed case
    most = max(33, min(0.4 * faces, 1.5e7 / edges ** 2, 30000))
    n = int(_log(rng, 32, most))
    if call == "step":
        kinds = ["nve", "abp"] if prec == "fp32" else ["nve", "bd", "abp", "gd", "fire"]
        more.update(dynamics=rng.choice(kinds), steps=rng.randint(1, 4))
        more["potential"] = "wca" if more["dynamics"] == "bd" else "harmonic"
    return _case("", call, surface, size, n, edges * edge, prec, **more)


# ------------------------------------------------------------------------------- surfaces

@functools.lru_cache(maxsize=12)
def _unit_sphere(level):
    t = (1.0 + 5 ** 0.5) / 2.0
    v = np.array([(-1, t, 0), (1, t, 0), (-1, -t, 0), (1, -t, 0), (0, -1, t), (0, 1, t), (0, -1, -t), (0, 1, -t),
                  (t, 0, -1), (t, 0, 1), (-t, 0, -1), (-t, 0, 1)], float)
    v /= np.linalg.norm(v, axis=1, keepdims=True)
    f = np.array([(0, 11, 5), (0, 5, 1), (0, 1, 7), (0, 7, 10), (0, 10, 11), (1, 5, 9), (5, 11, 4), (11, 10, 2),
                  (10, 7, 6), (7, 1, 8), (3, 9, 4), (3, 4, 2), (3, 2, 6), (3, 6, 8), (3, 8, 9), (4, 9, 5), (2, 4, 11),
                  (6, 2, 10), (8, 6, 7), (9, 8, 1)], np.int64)
    for _ in range(level):
        nv, nf = len(v), len(f)
        e = np.concatenate([f[:, [0, 1]], f[:, [1, 2]], f[:, [2, 0]]])
        lo, hi = e.min(axis=1), e.max(axis=1)
        key, inv = np.unique(lo * nv + hi, return_inverse=True)
        mid = v[key // nv] + v[key % nv]
        v = np.concatenate([v, mid / np.linalg.norm(mid, axis=1, keepdims=True)])
        m = nv + inv.reshape(3, nf)
        f = np.concatenate([np.stack([f[:, 0], m[0], m[2]], 1), np.stack([f[:, 1], m[1], m[0]], 1),
                            np.stack([f[:, 2], m[2], m[1]], 1), np.stack([m[0], m[1], m[2]], 1)])
    return v, np.ascontiguousarray(f, np.int32)


def _quads(nu, nv, wrap):
    """Two triangles for every cell of an nu x nv vertex grid (index i * nv + j)."""
    i, j = np.meshgrid(np.arange(nu if wrap else nu - 1), np.arange(nv if wrap else nv - 1), indexing="ij")
    at = lambda a, b: ((a % nu) * nv + b % nv).ravel()  # noqa: E731
    a, b, c, d = at(i, j), at(i + 1, j), at(i, j + 1), at(i + 1, j + 1)
    return np.ascontiguousarray(np.stack([np.stack([a, b, d], 1), np.stack([a, d, c], 1)], 1).reshape(-1, 3), np.int32)


def _torus(faces, major, minor):
    n_v = max(3, int(round(math.sqrt(faces / 2.0 * minor / major))))
    n_u = max(3, int(round(faces / (2.0 * n_v))))
    u, w = np.meshgrid(2 * np.pi * np.arange(n_u) / n_u, 2 * np.pi * np.arange(n_v) / n_v, indexing="ij")
    x = np.stack([(major + minor * np.cos(w)) * np.cos(u), (major + minor * np.cos(w)) * np.sin(u), minor * np.sin(w)],
                 -1).reshape(-1, 3)
    return x, _quads(n_u, n_v, True), None


def _surface(case, rng):
    """(vertices, faces, period or None)"""
    kind, size = case["surface"], case["size"]
    if kind == "sphere":
        v, f = _unit_sphere(size)
        r = case["scale"] + case["noise"] * rng.standard_normal(len(v))
        return v * r[:, None], f, None
    if kind == "torus":
        return _torus(size, case["aspect"], 1.0)
    if kind == "heightfield":   # a sum of periodic bumps over the unit square
        g = np.arange(size) / size
        x, y = np.meshgrid(g, g, indexing="ij")
        z = np.zeros_like(x)
        for amp, w, (cx, cy) in zip(rng.uniform(0.05, 0.3, 32), rng.uniform(0.05, 0.2, 32), rng.uniform(0, 1, (32, 2))):
            gx = sum(np.exp(-(g - cx - s) ** 2 / (2 * w * w)) for s in (-1, 0, 1))
            gy = sum(np.exp(-(g - cy - s) ** 2 / (2 * w * w)) for s in (-1, 0, 1))
            z += amp * np.outer(gx, gy)
        return np.stack([x, y, z], -1).reshape(-1, 3), _quads(size, size, True), (1.0, 1.0)
    g = np.linspace(0.0, 1.0, size)
    x, y = np.meshgrid(g, g, indexing="ij")
    return np.stack([x, y, 0 * x], -1).reshape(-1, 3), _quads(size, size, False), None


def _corners(verts, faces, period):
    p = verts[faces]
    if period is not None:
        for ax, length in enumerate(period):
            for k in (1, 2):
                p[:, k, ax] -= length * np.round((p[:, k, ax] - p[:, 0, ax]) / length)
    return p


def _scatter(verts, faces, period, n, rng):
    """n particles, uniform by area: faces, barycentrics, unit face normals."""
    p = _corners(verts, faces, period)
    nrm = np.cross(p[:, 1] - p[:, 0], p[:, 2] - p[:, 0])
    area = np.linalg.norm(nrm, axis=1)
    cdf = np.cumsum(area)
    face = np.minimum(np.searchsorted(cdf, rng.uniform(0, cdf[-1], n)), len(faces) - 1).astype(np.int32)
    r, u = np.sqrt(rng.uniform(0, 1, n)), rng.uniform(0, 1, n)
    bary = np.clip(np.stack([1 - r, r * (1 - u), r * u], 1), 1e-6, None)
    return face, bary / bary.sum(1, keepdims=True), nrm[face] / area[face, None]


def _tangent(normal, rng, unit):
    v = rng.standard_normal(normal.shape)
    v -= np.sum(v * normal, 1, keepdims=True) * normal
    return v / np.linalg.norm(v, axis=1, keepdims=True) if unit else v * math.sqrt(0.1)


def _potential(case):
    rc = case["reach"]
    kind = case["potential"]
    sigma = {"harmonic": rc, "wca": rc / 2.0 ** (1.0 / 6.0), "gaussian": rc / 3.0}[kind]
    return dict(kind=POTENTIALS[kind], eps=1.0, sigma=sigma, r_cut=rc, A=1.0)


def _integrator(case):
    kind = case["dynamics"]
    return dict(kind=DYNAMICS[kind], dt={"nve": 0.002, "bd": 1e-5, "abp": 1e-3, "gd": 1e-4, "fire": 1e-3}[kind],
                kT=1.0 if kind == "bd" else 0.1, lam=1.0, v0=1.0 if kind == "abp" else 0.0,
                Dr=0.1 if kind == "abp" else 0.0, mass=1.0,
                max_disp=0.5 * case["reach"] if kind in ("bd", "abp", "gd") else math.inf)


def _capacity(case):
    """Length of the program's pair table: half as much again as uniform particles need."""
    n, rc = case["particles"], case["reach"]
    if rc == 0:
        return n * (n - 1)
    need = n * (n - 1) * min(1.0, math.pi * rc * rc / _extent(case)[1])
    return int(max(16, 0.6 * min(64, n) / n * need)) if case["call"] == "paths" else int(1.5 * need) + 4 * n + 64


def _extent(case):
    """(faces, area) of the surface, about."""
    size = case["size"]
    return {"sphere": (20 * 4 ** size, 4 * math.pi * case["scale"] ** 2), "torus": (size, 4 * math.pi ** 2 * case["aspect"]),
            "heightfield": (2 * size * size, 1.3), "plane": (2 * (size - 1) ** 2, 1.0)}[case["surface"]]


def _table(rows, j, dist, tangent, capacity):
    """The rows in the program's own table of fixed length (unused entries zero)."""
    k = len(j)
    tj, td, tt = np.zeros(capacity, np.int32), np.zeros(capacity), np.zeros((capacity, 3))
    tj[:k], td[:k], tt[:k] = j, dist, tangent
    return {"rows": rows, "j": tj, "dist": td, "tangent": tt}


def _inputs(case, seed):
    """Host inputs of a case: a list of (verts, faces, period, face, bary, vel, orient)."""
    out = []
    for k in range(case["sets"]):
        rng = np.random.default_rng([seed, k])
        if case["call"] == "batch":   # tori of 2k-60k faces and 128-4096 particles, sizes fixed by the set's number
            fixed = np.random.default_rng(4000 + k)
            nf, n = int(math.exp(fixed.uniform(math.log(2000), math.log(60000)))), int(fixed.integers(128, 4097))
            v, f, per = _torus(nf, fixed.uniform(1.0, 3.0), fixed.uniform(0.3, 0.9))
        else:
            v, f, per = _surface(case, rng)
            n = case["particles"]
        face, bary, normal = _scatter(v, f, per, n, rng)
        vel = _tangent(normal, rng, False) if case["dynamics"] in ("nve", "fire") else None
        orient = _tangent(normal, rng, True) if case["dynamics"] == "abp" else None
        out.append((v, f, per, face, bary, vel, orient))
    return out


class _State:
    """What the program holds; frees the library's objects with itself."""

    def __init__(self):
        self.ctx = css.create(0)
        self.meshes, self.parts, self.batch = [], [], None

    def __del__(self):
        if self.batch is not None:
            self.batch.free()
        for x in self.parts + self.meshes:
            x.free()
        self.ctx.close()


def prepare(case, seed):
    s = _State()
    s.case = case
    s.prec = css.FP32 if case["precision"] == "fp32" else css.FP64
    s.r_c = case["reach"] if case["reach"] > 0 else math.inf
    s.start = []
    for v, f, per, face, bary, vel, orient in _inputs(case, seed):
        mesh = css.mesh_upload(s.ctx, v, f, per)
        s.meshes.append(mesh)
        s.parts.append(css.particles_set(s.ctx, mesh, face, bary, vel, orient, seed=seed))
        # the state a host loop feeds in each pass, and the buffers it reads back into
        s.start.append([None if a is None else torch.from_numpy(np.ascontiguousarray(a)).to(DEV)
                        for a in (face, bary, vel, orient)])
    call = case["call"]
    if call in ("forces", "step", "batch") and case["reach"] > 0:
        s.pot = _potential(case)
    if call in ("step", "batch"):
        s.integ = _integrator(case)
    if call == "batch":
        s.batch = css.batch_create(s.ctx, s.parts)
    s.out = [[torch.empty(len(p[0]), dtype=torch.int32, device=DEV)] +
             [torch.empty(len(p[0]), 3, dtype=torch.float64, device=DEV) for _ in range(4)] for p in s.start]
    s.pairs = _capacity(case)
    if call == "paths":   # neighbours of the first particles, as many pairs for every seed
        rs, j, _, _ = css.geodesic_neighbors(s.parts[0], s.r_c, css.FP64)
        src, dst = np.repeat(np.arange(len(rs) - 1), np.diff(rs)), j
        if len(src) < s.pairs:
            src, dst = np.resize(np.r_[src, 0], s.pairs), np.resize(np.r_[dst, 1], s.pairs)
        s.src, s.dst = src[:s.pairs].astype(np.int32), dst[:s.pairs].astype(np.int32)
    torch.cuda.synchronize()
    return s


def _real(s, x):
    """A real result in the precision the program keeps it in."""
    if s.prec == css.FP64:
        return x
    return x.float() if isinstance(x, torch.Tensor) else np.float32(x)


def run(s):
    call, case = s.case["call"], s.case
    if call == "forces":
        force, energy = css.compute_forces(s.parts[0], s.pot, s.r_c, s.prec, out=s.out[0][4])
        return {"force": _real(s, force), "energy": _real(s, energy)}
    if call == "neighbors":
        return _table(*css.geodesic_neighbors(s.parts[0], s.r_c, s.prec, capacity=s.pairs), s.pairs)
    if call == "vhm":
        return _table(*css.vhm_neighbors(s.parts[0], s.r_c, capacity=s.pairs), s.pairs)
    if call == "paths":
        points, legs, dist, _ = css.geodesic_paths(s.parts[0], s.r_c, s.src, s.dst, max_points=64)
        table = np.zeros((s.pairs, 64, 3))
        for k, p in enumerate(points):
            table[k, :len(p)] = p
        return {"points": table, "legs": legs, "dist": dist}
    # a host-driven loop: write the state in, advance it, read it back
    for p, (face, bary, vel, orient) in zip(s.parts, s.start):
        css.particles_update(p, face, bary, vel, orient)
        if case["dynamics"] in ("bd", "abp"):
            css.particles_set_step(p, 0)
    if call == "batch":
        css.batch_step(s.batch, s.pot, s.integ, s.r_c, s.prec, case["steps"])
    else:
        css.integrate_step(s.parts[0], s.pot, s.integ, s.r_c, s.prec, case["steps"])
    res = []
    for p, (face, bary, vel, orient, force) in zip(s.parts, s.out):
        css.particles_get_into(p, face, bary, vel, orient, force)
        res.append({"face": face, "bary": _real(s, bary), "force": _real(s, force)})
        if case["dynamics"] in ("nve", "fire"):
            res[-1]["vel"] = _real(s, vel)
        if case["dynamics"] == "abp":
            res[-1]["orient"] = _real(s, orient)
    return res


def work(case):
    """Bytes: the mesh records in reach, the particles and the outputs, each once.  Operations: about
    150 for each unfolding (two for each face in reach of a source), 20 for each pair; the
    approximate solver: one multiply-add per entry of a row for about sqrt(faces) sweeps."""
    nbytes = flops = 0.0
    for k in range(case["sets"]):
        if case["call"] == "batch":
            fixed = np.random.default_rng(4000 + k)
            nf, n = int(math.exp(fixed.uniform(math.log(2000), math.log(60000)))), int(fixed.integers(128, 4097))
            area = 4 * math.pi ** 2 * fixed.uniform(1.0, 3.0) * fixed.uniform(0.3, 0.9)
        else:
            n = case["particles"]
            nf, area = _extent(case)
        rc = case["reach"]
        part = min(1.0, math.pi * rc * rc / area) if rc > 0 else 1.0
        near, pairs = max(3.0, part * nf), n * (n - 1) * part
        sources = min(64, n) if case["call"] == "paths" else n
        pairs *= sources / n
        nbytes += min(nf, sources * near) * 192 + n * 28
        if case["call"] == "vhm":
            flops += n * nf / 2 * 7 * 2 * 4 * math.sqrt(nf)
            nbytes += pairs * 36
        else:
            steps = case["steps"] + (1 if case["dynamics"] in ("nve", "fire") else 0)
            flops += steps * (sources * 2 * near * 150 + pairs * 20)
            nbytes += pairs * 36 if case["call"] in ("neighbors", "paths") else n * 124
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------------------- 64-bit values

def _expand(count):
    """(owner, rank within the owner) of every item of a ragged list with these counts."""
    owner = torch.repeat_interleave(torch.arange(len(count), device=count.device), count)
    first = torch.cumsum(count, 0) - count
    return owner, torch.arange(len(owner), device=count.device) - first[owner]


class _Polyhedron:
    """Half-edge geometry and straight rays on a triangulated surface (64-bit torch)."""

    def __init__(self, verts, faces, period):
        f = torch.from_numpy(faces.astype(np.int64)).to(DEV)
        p = torch.from_numpy(np.ascontiguousarray(_corners(verts, faces, period))).to(DEV)
        self.nf, nv = len(f), len(verts)
        u, v = f.reshape(-1), f[:, [1, 2, 0]].reshape(-1)
        key, back = u * nv + v, v * nv + u
        order = torch.argsort(key)
        at = torch.searchsorted(key[order], back).clamp(max=len(key) - 1)
        hit = key[order][at] == back
        self.twin = torch.where(hit, order[at], torch.full_like(at, -1))
        self.u, self.v, self.c = u, v, f[:, [2, 0, 1]].reshape(-1)
        side = (p[:, [1, 2, 0]] - p).norm(dim=2)              # lengths of the half-edges
        self.L = side.reshape(-1)
        b, a = side[:, [2, 0, 1]].reshape(-1), side[:, [1, 2, 0]].reshape(-1)
        self.cx = (self.L ** 2 + b ** 2 - a ** 2) / (2 * self.L)
        self.cy = (b ** 2 - self.cx ** 2).clamp(min=0).sqrt()
        ang = torch.atan2(self.cy, self.cx)
        theta = torch.zeros(nv, dtype=torch.float64, device=DEV).index_add_(0, u, ang)
        rim = torch.zeros(nv, dtype=torch.bool, device=DEV)
        rim[u[~hit]] = True
        rim[v[~hit]] = True
        bend = torch.where(rim, theta > math.pi + 1e-10, theta > 2 * math.pi + 1e-10)
        self.saddle = torch.nonzero(bend).reshape(-1)         # where shortest paths may bend
        self.slot = torch.full((nv,), -1, dtype=torch.int64, device=DEV)
        self.slot[self.saddle] = torch.arange(len(self.saddle), device=DEV)
        e1 = (p[:, 1] - p[:, 0]) / side[:, 0:1]
        e2 = p[:, 2] - p[:, 0]
        e2 = e2 - (e2 * e1).sum(1, keepdim=True) * e1
        self.e1, self.e2 = e1, e2 / e2.norm(dim=1, keepdim=True)

    def local(self, face, bary):
        h = 3 * face
        return (bary[:, 1] * self.L[h] + bary[:, 2] * self.cx[h], bary[:, 2] * self.cy[h])

    def frame(self, h, x, y):
        """A point of the face's layout in the frame of half-edge h (origin its start, x along it)."""
        k, h0 = h % 3, h - h % 3
        L, cx, cy = self.L[h0], self.cx[h0], self.cy[h0]
        zero = torch.zeros_like(L)
        ax = torch.where(k == 0, zero, torch.where(k == 1, L, cx))
        ay = torch.where(k == 2, cy, zero)
        bx = torch.where(k == 0, L, torch.where(k == 1, cx, zero))
        by = torch.where(k == 1, cy, zero)
        dx, dy = (bx - ax) / self.L[h], (by - ay) / self.L[h]
        return (x - ax) * dx + (y - ay) * dy, dx * (y - ay) - dy * (x - ax), dx, dy

    def rays(self, node, h, sx, sy, ta, tb, rc, first, items, tx, ty):
        """Straight lines from points s seen through whole half-edges h, within rc.  Yields what they
        reach: (node, vertex, length, direction) and (node, target, length, direction); a direction
        is written in the axes whose image is (ta, tb)."""
        b0, b1 = torch.zeros_like(sx), self.L[h]
        for _ in range(100000):
            if len(h) == 0:
                return
            L, cx, cy = self.L[h], self.cx[h], self.cy[h]
            f = h // 3
            own, k = _expand(first[f + 1] - first[f])
            if len(own):
                j = items[first[f[own]] + k]
                hx, hy, _, _ = self.frame(h[own], tx[j], ty[j])
                dx, dy = hx - sx[own], hy - sy[own]
                at = sx[own] + dx * -sy[own] / dy
                d = (dx * dx + dy * dy).sqrt()
                ok = (at >= b0[own] - 1e-12 * L[own]) & (at <= b1[own] + 1e-12 * L[own]) & (d < rc)
                o, d = own[ok], d[ok]
                cs, sn = dx[ok] / d, dy[ok] / d
                yield "target", node[o], j[ok], d, cs * ta[o] + sn * tb[o], -cs * tb[o] + sn * ta[o]
            dx, dy = cx - sx, cy - sy
            xc = sx + dx * -sy / dy
            d = (dx * dx + dy * dy).sqrt()
            c = self.c[h]
            ok = (xc >= b0 - 1e-12 * L) & (xc <= b1 + 1e-12 * L) & (d < rc) & (self.slot[c] >= 0)
            if ok.any():
                cs, sn = dx[ok] / d[ok], dy[ok] / d[ok]
                yield "vertex", node[ok], self.slot[c[ok]], d[ok], cs * ta[ok] + sn * tb[ok], -cs * tb[ok] + sn * ta[ok]
            parts = []
            for side in (0, 1):
                across = h - h % 3 + (h + (2 if side == 0 else 1)) % 3
                tw = self.twin[across]
                go = (tw >= 0) & ((xc > b0) if side == 0 else (xc < b1))
                i = torch.nonzero(go).reshape(-1)
                zero = torch.zeros_like(L[i])
                ax, ay = (zero, zero) if side == 0 else (cx[i], cy[i])
                ex, ey = (cx[i], cy[i]) if side == 0 else (L[i] - cx[i], -cy[i])
                le = (ex * ex + ey * ey).sqrt()

                def cut(X):
                    rx, ry = X - sx[i], -sy[i]
                    return (((sx[i] - ax) * ry - (sy[i] - ay) * rx) / (ex * ry - ey * rx)).clamp(0, 1) * le
                if side == 0:
                    n0, n1 = cut(b0[i]), torch.where(b1[i] >= xc[i], le, cut(b1[i]))
                else:
                    n0, n1 = torch.where(b0[i] <= xc[i], zero, cut(b0[i])), cut(b1[i])
                co, si = ex / le, ey / le
                px, py = sx[i] - ax, sy[i] - ay
                qx, qy = px * co + py * si, (-px * si + py * co).clamp(max=0)
                near = torch.minimum(torch.maximum(qx, n0), n1) - qx
                keep = (n1 - n0 > 1e-12 * le) & ((near * near + qy * qy).sqrt() < rc)
                parts.append([t[keep] for t in (node[i], tw[i], qx, qy, ta[i] * co + tb[i] * si,
                                                -ta[i] * si + tb[i] * co, n0, n1)])
            node, h, sx, sy, ta, tb, b0, b1 = (torch.cat(t) for t in zip(*parts))

    def reach(self, start, rc, first, items, tx, ty):
        """All that straight lines from the start windows reach, one row for each (node, goal): the shortest."""
        got = {"target": [], "vertex": []}
        for r in self.rays(*start, rc, first, items, tx, ty):
            got[r[0]].append(r[1:])
        return {k: [torch.cat(t) for t in zip(*v)] if v else None for k, v in got.items()}


def _shortest(a, b, d, ex, ey, nb):
    """One row for each (a, b), the shortest, sorted by a and then b."""
    o = torch.argsort(d, stable=True)
    o = o[torch.argsort((a * nb + b)[o], stable=True)]
    key = (a * nb + b)[o]
    lead = torch.ones_like(key, dtype=torch.bool)
    lead[1:] = key[1:] != key[:-1]
    o = o[lead]
    return a[o], b[o], d[o], ex[o], ey[o]


def _pairs(verts, faces, period, face, bary, rc):
    """All ordered pairs closer than rc: (i, j, length, world direction at i), sorted."""
    m = _Polyhedron(verts, faces, period)
    n = len(face)
    fc, bc = torch.from_numpy(face.astype(np.int64)).to(DEV), torch.from_numpy(bary).to(DEV)
    tx, ty = m.local(fc, bc)
    items = torch.argsort(fc, stable=True)
    first = torch.zeros(m.nf + 1, dtype=torch.int64, device=DEV)
    first[1:] = torch.cumsum(torch.bincount(fc, minlength=m.nf), 0)
    ns = len(m.saddle)
    found, vert = [], []
    per = 40000
    for lo in range(0, n, per):   # straight from the particles
        i = torch.arange(lo, min(lo + per, n), device=DEV)
        own, k = _expand(first[fc[i] + 1] - first[fc[i]])   # the source's own face
        j = items[first[fc[i[own]]] + k]
        ok = j != i[own]
        a, j = i[own][ok], j[ok]
        dx, dy = tx[j] - tx[a], ty[j] - ty[a]
        d = (dx * dx + dy * dy).sqrt()
        found.append((a, j, d, dx / d, dy / d))
        corner = torch.arange(3, device=DEV).repeat(len(i))
        ii = i.repeat_interleave(3)
        h = 3 * fc[ii] + corner
        hx, hy, dx, dy = m.frame(h, tx[ii], ty[ii])
        s = m.slot[m.u[h]]
        ok = s >= 0
        if ok.any():   # its own corners: the direction from the particle to the edge's start
            d = (hx[ok] ** 2 + hy[ok] ** 2).sqrt()
            vx, vy = -hx[ok] / d, -hy[ok] / d
            vert.append((ii[ok], s[ok], d, vx * dx[ok] - vy * dy[ok], vx * dy[ok] + vy * dx[ok]))
        tw = m.twin[h]
        ok = tw >= 0
        r = m.reach((ii[ok], tw[ok], (m.L[h] - hx)[ok], (-hy)[ok], -dx[ok], dy[ok]), rc, first, items, tx, ty)
        if r["target"]:
            found.append(r["target"])
        if r["vertex"]:
            vert.append(r["vertex"])
    if ns and vert:
        # straight from the saddle vertices, through the edge opposite each of their corners
        corners = torch.nonzero(m.slot[m.u] >= 0).reshape(-1)
        hop, link = [], []
        per = 120000
        for lo in range(0, len(corners), per):
            h = corners[lo:lo + per]
            node, f = m.slot[m.u[h]], h // 3
            own, k = _expand(first[f + 1] - first[f])
            if len(own):
                j = items[first[f[own]] + k]
                hx, hy, _, _ = m.frame(h[own], tx[j], ty[j])
                hop.append((node[own], j, (hx * hx + hy * hy).sqrt()))
            for goal, d in ((m.v[h], m.L[h]), (m.c[h], (m.cx[h] ** 2 + m.cy[h] ** 2).sqrt())):
                ok = m.slot[goal] >= 0
                link.append((node[ok], m.slot[goal[ok]], d[ok]))
            e = h - h % 3 + (h + 1) % 3
            tw = m.twin[e]
            ok = tw >= 0
            one = torch.ones_like(m.L[e][ok])
            r = m.reach((node[ok], tw[ok], (m.L[e] - m.cx[e])[ok], (-m.cy[e])[ok], one, 0 * one), rc, first, items, tx, ty)
            if r["target"]:
                hop.append(r["target"][:3])
            if r["vertex"]:
                link.append(r["vertex"][:3])
        zero = lambda t: (t, torch.zeros_like(t), torch.zeros_like(t))  # noqa: E731
        la, lb, ld, _, _ = _shortest(*(torch.cat(t) for t in list(zip(*link))[:2]), *zero(torch.cat([x[2] for x in link])), ns)
        ha, hj, hd, _, _ = _shortest(*(torch.cat(t) for t in list(zip(*hop))[:2]), *zero(torch.cat([x[2] for x in hop])), n)
        ok = ld < rc
        la, lb, ld = la[ok], lb[ok], ld[ok]
        lfirst = torch.searchsorted(la, torch.arange(ns + 1, device=DEV))
        hfirst = torch.searchsorted(ha, torch.arange(ns + 1, device=DEV))
        va, vb, vd, vx, vy = _shortest(*(torch.cat(t) for t in zip(*vert)), ns)
        chunk = max(1, min(n, 200_000_000 // (8 * ns)))
        for lo in range(0, n, chunk):   # chains of saddle vertices, a block of sources at a time
            a, b = torch.searchsorted(va, torch.tensor([lo, lo + chunk], device=DEV)).tolist()
            best = torch.full((chunk * ns,), math.inf, dtype=torch.float64, device=DEV)
            ex, ey = torch.zeros_like(best), torch.zeros_like(best)
            at = (va[a:b] - lo) * ns + vb[a:b]
            best[at], ex[at], ey[at] = vd[a:b], vx[a:b], vy[a:b]
            live = at
            while len(live):
                new = []
                for part in live.split(200000):
                    s = part % ns
                    own, k = _expand(lfirst[s + 1] - lfirst[s])
                    e = lfirst[s[own]] + k
                    src, to = part[own], part[own] - s[own] + lb[e]
                    d = best[src] + ld[e]
                    ok = (d < rc) & (d < best[to] - 1e-14)
                    src, to, d = src[ok], to[ok], d[ok]
                    if not len(to):
                        continue
                    best.scatter_reduce_(0, to, d, "amin")
                    won = best[to] == d
                    ex[to[won]], ey[to[won]] = ex[src[won]], ey[src[won]]
                    new.append(to[won])
                live = torch.unique(torch.cat(new)) if new else live[:0]
            full = torch.nonzero(best < rc).reshape(-1)
            for part in full.split(400000):
                s = part % ns
                own, k = _expand(hfirst[s + 1] - hfirst[s])
                e = hfirst[s[own]] + k
                d = best[part[own]] + hd[e]
                ok = d < rc
                o, e, d = part[own[ok]], e[ok], d[ok]
                found.append((lo + torch.div(o, ns, rounding_mode="floor"), hj[e], d, ex[o], ey[o]))
    i, j, d, x, y = _shortest(*(torch.cat(t) for t in zip(*found)), n)
    ok = (d < rc) & (i != j)
    i, j, d, x, y = i[ok], j[ok], d[ok], x[ok], y[ok]
    t = x[:, None] * m.e1[fc[i]] + y[:, None] * m.e2[fc[i]]
    return i, j, d, t


def _force(pot, i, d, t, n):
    eps, sg, A = pot["eps"], pot["sigma"], pot["A"]
    if pot["kind"] == css.POT_HARMONIC:
        u, du = eps * (1 - d / sg) ** 2, -2 * eps * (1 - d / sg) / sg
    elif pot["kind"] == css.POT_WCA:
        q6 = (sg / d) ** 6
        u, du = 4 * eps * (q6 * q6 - q6) + eps, 24 * eps * (q6 - 2 * q6 * q6) / d
    else:
        u = A * torch.exp(-d * d / (2 * sg * sg))
        du = -d / (sg * sg) * u
    near = d < pot["r_cut"]
    u, du = torch.where(near, u, 0 * u), torch.where(near, du, 0 * du)
    return torch.zeros(n, 3, dtype=torch.float64, device=DEV).index_add_(0, i, du[:, None] * t), float(0.5 * u.sum())


def exact(case, seed):
    call, rc = case["call"], case["reach"] if case["reach"] > 0 else math.inf
    if call in ("vhm", "paths", "batch"):   # an iterative approximation; polylines; several moves
        return None
    if call == "step" and (case["steps"] != 1 or case["dynamics"] in ("nve", "fire")):
        return None
    if call == "neighbors" and case["surface"] == "torus" and rc == math.inf:
        return None    # rays that nothing trims grow too many over a whole torus
    v, f, per, face, bary, _, _ = _inputs(case, seed)[0]
    i, j, d, t = _pairs(v, f, per, face, bary, rc)
    n = len(face)
    if call == "neighbors":
        rows = torch.searchsorted(i, torch.arange(n + 1, device=DEV))
        return _table(rows.cpu().numpy(), j.to(torch.int32).cpu().numpy(), d.cpu().numpy(), t.cpu().numpy(), _capacity(case))
    force, energy = _force(_potential(case), i, d, t, n)
    if call == "forces":
        return {"force": force, "energy": energy}
    # one overdamped step moves the particles along the force at its start; the move has no plain form here
    out = {"face": None, "bary": None, "force": force}
    if case["dynamics"] == "abp":
        out["orient"] = None
    return [out]
