"""The neighbour kernel where its working memory ends and where a source is degenerate (needs a
GB300).  FP64 distances equal the oracle's to 1e-9 (the bar of the parity tests); launch shapes
that overflow the ring, the vertex table or the target table give the same pairs."""
import math

import numpy as np
import pytest

import synth
from oracle import oracle as O
from tests._common import FP32_REL_DIAM, FP64_RTOL, compare_pairs, sample_sources, select_rows

css = pytest.importorskip("paper_2404_19751_gb300")
pytestmark = pytest.mark.gpu

BASE = dict(warps_per_cta=4, ctas_per_sm=0, tile=1, shared_scale=1, window_capacity=2048,
            window_capacity2=16384, warps2_per_sm=2, occupancy=1, table_capacity=0, team=0)


@pytest.fixture(scope="module")
def ctx():
    c = css.create(0)
    yield c
    c.close()


def _rows(ctx, m, face, bary, r_c, prec=css.FP64, **shape):
    before = ctx.get_launch()
    ctx.set_launch(**dict(BASE, **shape))
    mesh = css.mesh_upload(ctx, m.verts, m.faces, m.period)
    parts = css.particles_set(ctx, mesh, face, bary)
    try:
        return css.geodesic_neighbors(parts, r_c, prec), ctx.last_counters()["deferred"]
    finally:
        ctx.set_launch(**before)
        parts.free()
        mesh.free()


# targets per source: around the shared table's fill (56 of 64), the rank sort's limit (128), the
# next powers of two, and beyond the second pass's first table (3584 of 4096)
@pytest.mark.parametrize("n,deferred", [(2, False), (56, False), (58, True), (129, True), (130, True), (258, True),
                                        (3700, True)])
def test_target_table_edges(ctx, n, deferred):
    m = synth.icosphere(1, 1.0, noise=0.1, seed=3)
    face, bary = synth.place_uniform(m, n, 5)
    g, d = _rows(ctx, m, face, bary, math.inf)
    assert (d > 0) == deferred
    assert np.all(np.diff(g[0]) == n - 1)
    want = np.tile(np.arange(n), (n, 1))[~np.eye(n, dtype=bool)]
    assert np.array_equal(g[1], want)
    src = sample_sources(n, 8, 2)
    compare_pairs(select_rows(g, src), O.OracleMesh(m).neighbors_gap(face, bary, math.inf, sources=src), math.inf,
                  FP64_RTOL, 1e-7)


SHAPES = [dict(window_capacity=64), dict(window_capacity=1024), dict(window_capacity=512, team=1, warps_per_cta=2),
          dict(team=1, warps_per_cta=8), dict(team=1, warps_per_cta=8, shared_scale=8, window_capacity=8192),
          dict(shared_scale=0, window_capacity=8192, table_capacity=512),
          dict(shared_scale=0, window_capacity=8192, table_capacity=512, team=1, warps_per_cta=3),
          dict(shared_scale=8, warps_per_cta=1, window_capacity=16384)]


@pytest.mark.parametrize("name", ["holed", "fan", "rough", "hfield"])
def test_overflowing_shapes_give_the_same_pairs(ctx, name):
    m, n, r_c = {"holed": (synth.holed_plane(21), 60, math.inf), "fan": (synth.saddle_fan(8, 6), 50, math.inf),
                 "rough": (synth.icosphere(4, 1.0, noise=0.03, seed=2), 200, 0.6),
                 "hfield": (synth.periodic_heightfield(48, 16, seed=4), 150, 0.3)}[name]
    face, bary = synth.place_uniform(m, n, 9)
    ref = O.OracleMesh(m).neighbors_gap(face, bary, r_c)
    base, _ = _rows(ctx, m, face, bary, r_c)
    compare_pairs(base, ref, r_c, FP64_RTOL, 1e-7)
    for sh in SHAPES:
        g, _ = _rows(ctx, m, face, bary, r_c, **sh)
        assert np.array_equal(g[0], base[0]) and np.array_equal(g[1], base[1]), sh
        np.testing.assert_allclose(g[2], base[2], rtol=1e-13, atol=0, err_msg=str(sh))


@pytest.mark.parametrize("team", [0, 1])
def test_sources_on_and_near_vertices(ctx, team):
    """Particles exactly on vertices (interior, boundary, saddle), on edges, and 1e-14 to 1e-3 of an
    edge away from a vertex: distances equal the oracle's in both forms."""
    for m, r_c in ((synth.icosphere(2, 1.0, noise=0.05, seed=6), 1.1), (synth.saddle_fan(8, 4), math.inf),
                   (synth.grid_plane(6, 6), 0.7), (synth.holed_plane(11), 0.6)):
        rng = np.random.default_rng(3)
        face, bary = synth.place_uniform(m, 48, 4)
        for k in range(36):
            eps = [0.0, 1e-14, 1e-12, 1e-9, 1e-6, 1e-3][k % 6]
            b = np.array([1.0 - 1.7 * eps, eps, 0.7 * eps])
            if k >= 30:
                b = np.array([0.0, 0.4, 0.6])
            bary[k] = np.roll(b, rng.integers(3))
        ref = O.OracleMesh(m).neighbors(face, bary, r_c)
        g, _ = _rows(ctx, m, face, bary, r_c, team=team, warps_per_cta=2)
        # distances below 1e-9 of an edge are compared absolutely
        ok = ref[2] > 1e-9
        assert np.array_equal(g[0], ref[0]) and np.array_equal(g[1], ref[1])
        np.testing.assert_allclose(g[2][ok], ref[2][ok], rtol=FP64_RTOL, atol=0)
        np.testing.assert_allclose(g[2][~ok], ref[2][~ok], rtol=FP64_RTOL, atol=7.2e-15)
        assert np.isfinite(g[3]).all()
        g32, _ = _rows(ctx, m, face, bary, r_c, css.FP32, team=team, warps_per_cta=2)
        tol = FP32_REL_DIAM * synth.bbox_diagonal(m)
        compare_pairs(g32, ref, r_c, tol, math.inf, rel=False, band=tol)   # at a vertex directions are set-valued
