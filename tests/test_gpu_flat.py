"""Large developable surfaces, where shortest paths have a closed form (needs a GB300).

Behind a flat vertex only the two straight windows beside it meet, so every gap between their
cones loses pairs or leaves a longer path.  Vertices are moved at random (within the surface):
on a regular grid the windows' edges lie on grid lines and round alike."""
import math

import numpy as np
import pytest

import synth
from synth.meshes import Mesh
from tests._common import FP32_REL_DIAM, FP64_RTOL

css = pytest.importorskip("paper_2404_19751_gb300")
pytestmark = pytest.mark.gpu


def _grid(u, v, wrap_u, wrap_v):
    """Triangles of an nu x nv vertex grid (index i * nv + j), two a cell."""
    nu, nv = u, v
    i, j = np.meshgrid(np.arange(nu if wrap_u else nu - 1), np.arange(nv if wrap_v else nv - 1), indexing="ij")
    at = lambda a, b: ((a % nu) * nv + b % nv).ravel()  # noqa: E731
    a, b, c, d = at(i, j), at(i + 1, j), at(i, j + 1), at(i + 1, j + 1)
    return np.stack([np.stack([a, b, d], 1), np.stack([a, d, c], 1)], 1).reshape(-1, 3).astype(np.int32)


def _surface(kind, n, seed):
    """A mesh of n x n vertices, their positions in the plane it unrolls to, and that plane's periods."""
    rng = np.random.default_rng(seed)
    if kind == "tube":   # a prism of n sides and perimeter 1; vertices move along its edges
        z = np.arange(n)[None, :] / n + np.zeros((n, 1))
        z[:, 1:-1] += rng.uniform(-0.15, 0.15, (n, n - 2)) / n
        phi = 2 * math.pi * np.arange(n)[:, None] / n + 0 * z
        rad = 1.0 / (2 * n * math.sin(math.pi / n))
        verts = np.stack([rad * np.cos(phi), rad * np.sin(phi), z], -1).reshape(-1, 3)
        flat = np.stack([np.arange(n)[:, None] / n + 0 * z, z], -1).reshape(-1, 2)
        return Mesh(verts, _grid(n, n, True, False)), flat, (1.0, 0.0)
    step = 1.0 / n if kind == "patch" else 1.0 / (n - 1)
    x, y = np.meshgrid(step * np.arange(n), step * np.arange(n), indexing="ij")
    flat = np.stack([x, y], -1).reshape(-1, 2)
    free = np.ones(n * n, bool) if kind == "patch" else (np.abs(flat - 0.5) < 0.5 - step / 2).all(1)
    flat[free] += rng.uniform(-0.15, 0.15, (free.sum(), 2)) * step
    if kind == "patch":
        flat %= 1.0
    verts = np.concatenate([flat, np.zeros((n * n, 1))], 1)
    wrap = kind == "patch"
    return Mesh(verts, _grid(n, n, wrap, wrap), (1.0, 1.0) if wrap else None), flat, (1.0, 1.0) if wrap else (0.0, 0.0)


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("kind,n,seed,edges", [("sheet", 80, 1, 0), ("sheet", 120, 2, 50), ("patch", 90, 1, 0),
                                               ("tube", 80, 1, 0), ("tube", 80, 20, 0)])
def test_every_pair_of_a_developable_surface(kind, n, seed, edges, prec):
    m, flat, period = _surface(kind, n, seed)
    count = 2500
    r_c = edges / n if edges else math.inf
    face, bary = synth.place_uniform(m, count, seed + 1)
    corner = flat[m.faces[face]].copy()
    for ax, p in enumerate(period):
        if p:
            corner[:, :, ax] -= np.round(corner[:, :, ax] - corner[:, :1, ax])
    x = np.einsum("nk,nkd->nd", bary, corner)
    d0 = x[None] - x[:, None]
    for ax, p in enumerate(period):
        if p:
            d0[:, :, ax] -= np.round(d0[:, :, ax])
    d0 = np.hypot(d0[:, :, 0], d0[:, :, 1])
    np.fill_diagonal(d0, np.inf)
    ctx = css.create(0)
    mesh = css.mesh_upload(ctx, m.verts, m.faces, m.period)
    parts = css.particles_set(ctx, mesh, face, bary)
    rs, j, d, _ = css.geodesic_neighbors(parts, r_c, getattr(css, prec.upper()))
    parts.free()
    mesh.free()
    ctx.close()
    got = np.full((count, count), np.inf)
    got[np.repeat(np.arange(count), np.diff(rs)), j] = d
    # the bars of the parity tests: relative in FP64, of the surface's size in FP32
    tol = FP64_RTOL * d0 if prec == "fp64" else np.full_like(d0, FP32_REL_DIAM * synth.bbox_diagonal(m))
    sure = np.isfinite(d0) & ((d0 < r_c - tol) if math.isfinite(r_c) else True)
    lost = sure & ~np.isfinite(got)
    assert not lost.any(), f"{lost.sum()} of {sure.sum()} pairs lost, first {np.argwhere(lost)[0]}"
    far = np.isfinite(got) & np.isfinite(d0)
    wrong = far & ~(np.abs(np.where(far, got, 0) - np.where(far, d0, 0)) <= tol)
    assert not wrong.any(), f"{wrong.sum()} lengths off, first {np.argwhere(wrong)[0]}"
    assert len(j) <= sure.sum() + (np.isfinite(d0) & ~sure & (d0 < r_c + tol)).sum()
