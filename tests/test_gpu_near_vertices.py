"""Sources and targets within rounding of vertices, and anywhere up to 1e-4 of an edge away, on flat sheets where
every distance is Euclidean (needs a GB300).  On a regular grid the lines from such a source to
such targets pass within rounding of the vertices between them."""
import math

import numpy as np
import pytest

import synth
from synth.particles import world_positions
from tests._common import FP32_REL_DIAM, FP64_RTOL

css = pytest.importorskip("paper_2404_19751_gb300")
pytestmark = pytest.mark.gpu

EPS = (0.0, 1e-16, 1e-15, 1e-14, 1e-13, 1e-12, 1e-11, 1e-10, 1e-9, 1e-8, 1e-7, 1e-6, 1e-4)


def _near_vertices(m, edges, rng):
    """20 particles for each offset, near a random corner of a random face: inside it, or on one of its edges."""
    n = 20 * len(EPS)
    face = rng.integers(0, m.nf, n).astype(np.int32)
    bary = np.zeros((n, 3))
    for k in range(n):
        u = 1.0 if edges else rng.uniform(0.1, 0.9)
        a, b = EPS[k // 20] * u, EPS[k // 20] * (1.0 - u)
        if edges:
            a *= rng.uniform(0.1, 1.0)
            if rng.random() < 0.5:
                a, b = b, a
        bary[k] = np.roll([1.0 - a - b, a, b], int(rng.integers(3)))
    return face, bary


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("moved", [0.0, 0.1])
@pytest.mark.parametrize("edges", [False, True])
def test_every_pair_next_to_vertices(edges, moved, prec):
    ctx = css.create(0)
    for seed in range(8):
        rng = np.random.default_rng(seed)
        m = synth.grid_plane(13, 13)
        v = m.verts.copy()
        inner = (np.abs(v[:, :2] - 0.5) < 0.49).all(1)
        v[inner, :2] += rng.uniform(-moved, moved, (inner.sum(), 2)) / 12
        m = synth.Mesh(v, m.faces, None)
        face, bary = _near_vertices(m, edges, rng)
        x = world_positions(m, face, bary)[:, :2]
        want = np.hypot(*(x[None] - x[:, None]).transpose(2, 0, 1))
        mesh = css.mesh_upload(ctx, m.verts, m.faces)
        parts = css.particles_set(ctx, mesh, face, bary)
        rs, j, d, _ = css.geodesic_neighbors(parts, math.inf, getattr(css, prec.upper()))
        parts.free()
        mesh.free()
        n = len(face)
        got = np.full((n, n), np.inf)
        got[np.repeat(np.arange(n), np.diff(rs)), j] = d
        np.fill_diagonal(got, 0.0)
        # positions are rounded to 1e-16 of the sheet on either side, distances near zero with them
        tol = FP64_RTOL * want + 1e-14 if prec == "fp64" else np.full((n, n), FP32_REL_DIAM * math.sqrt(2.0))
        bad = ~(np.abs(np.where(np.isfinite(got), got, 1e9) - want) <= tol)
        assert not bad.any(), f"seed {seed}: {bad.sum()} of {n * n} pairs, {np.isinf(got).sum()} of them lost, first {np.argwhere(bad)[0]}"
    ctx.close()
