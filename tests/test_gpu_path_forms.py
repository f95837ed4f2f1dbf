"""Shortest-path polylines by the path form's three routes: tables in shared memory, sources that
overflow them and are taken over, tables in global memory from the start; with a source on a
vertex.  Distances against the oracle to the FP64 form's 1e-9; every polyline as long as its
distance and landing on its nodes within 1e-9, the other path tests' tolerances (needs a GB300)."""
import math

import numpy as np
import pytest

import synth
from oracle import oracle as O

css = pytest.importorskip("paper_2404_19751_gb300")
pytestmark = pytest.mark.gpu


def _particles(m, n, crowd, seed):
    """n particles, the first `crowd` of them within a few edges of one vertex, particle 0 on it."""
    rng = np.random.default_rng(seed)
    v, f = np.asarray(m.verts), np.asarray(m.faces)
    c = v[f].mean(1)
    near = np.argsort(np.linalg.norm(c - c[5], axis=1))[:24]
    face = np.concatenate([rng.choice(near, crowd), rng.integers(0, len(f), n - crowd)]).astype(np.int32)
    bary = rng.dirichlet((2.0, 2.0, 2.0), n)
    face[0] = 5
    bary[0] = (0.0, 1.0, 0.0)
    return face, bary


@pytest.mark.parametrize("name,n,crowd,r_c", [("shared", 300, 1, 0.2), ("taken_over", 300, 200, 0.2),
                                              ("global", 40, 1, math.inf)])
def test_path_routes_match_oracle(name, n, crowd, r_c):
    m = synth.icosphere(4, 1.0, noise=0.02, seed=6)
    face, bary = _particles(m, n, crowd, 8)
    om = O.OracleMesh(m)
    src = np.arange(6, dtype=np.int32)
    rs, j = om.neighbors(face, bary, r_c, sources=src)[:2]
    S = np.repeat(src, np.diff(rs)).astype(np.int32)
    D = j.astype(np.int32)
    ctx = css.create(0)
    mesh = css.mesh_upload(ctx, m.verts, m.faces, m.period)
    parts = css.particles_set(ctx, mesh, face, bary)
    pts, legs, dist, gap = css.geodesic_paths(parts, r_c, S, D, max_points=2048)
    deferred = ctx.last_counters()["deferred"]
    ref = om.geodesic_paths(face, bary, r_c, S, D, cap=2048)[2]
    parts.free()
    mesh.free()
    ctx.close()
    assert (deferred > 0) == (name == "taken_over")
    np.testing.assert_allclose(dist, ref, rtol=1e-9, atol=0)
    assert np.all(legs >= 1) and gap.max() < 1e-9
    for p, d in zip(pts, dist):
        assert np.linalg.norm(np.diff(p, axis=0), axis=1).sum() == pytest.approx(d, rel=1e-9)
