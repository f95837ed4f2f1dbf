"""Shapes that a context picks by itself (needs a GB300): what one mesh or cutoff taught them does not carry
over to others, and the counters of other calls do not steer them."""
import numpy as np
import pytest

import synth

css = pytest.importorskip("paper_2404_19751_gb300")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def graded():
    """The unit square, spacings growing twentyfold along both axes; as many particles in a small face as in
    a large one, so that patches in the fine corner hold far more faces than their share of the area."""
    n = 64
    x = np.concatenate([[0.0], np.cumsum(20.0 ** (np.arange(n - 1) / (n - 2.0)))])
    m = synth.grid_plane(n, n)
    k = np.arange(n * n)
    v = np.stack([x[k % n], x[k // n], 0.0 * k], 1) / x[-1]
    m = synth.Mesh(v, m.faces, None)
    return (m,) + synth.place_uniform(m, 3000, 6, area_weighted=False)


def _deferred(ctx, parts, r_c):
    css.geodesic_neighbors(parts, r_c, css.FP64)
    return ctx.last_counters()["deferred"]


def test_larger_tables_stay_with_the_mesh_and_the_reach(graded):
    m, face, bary = graded
    near, far = 0.03, 0.05   # 22 and 62 faces by share of the area
    first = {}
    for r_c in (near, far):
        ctx = css.create(0)
        mesh = css.mesh_upload(ctx, m.verts, m.faces)
        parts = css.particles_set(ctx, mesh, face, bary)
        first[r_c] = _deferred(ctx, parts, r_c)
        assert first[r_c] * 25 > len(face)
        if r_c == near:   # tables grow until few sources are deferred
            later = [_deferred(ctx, parts, r_c) for _ in range(6)]
            assert later[-1] * 25 <= len(face), later
            mesh2 = css.mesh_upload(ctx, m.verts, m.faces)
            parts2 = css.particles_set(ctx, mesh2, face, bary)
            assert _deferred(ctx, parts2, r_c) == first[r_c]
            other = _deferred(ctx, parts, far)
            parts2.free()
            mesh2.free()
        parts.free()
        mesh.free()
        ctx.close()
    assert other == first[far]


def test_only_deferrals_bring_the_second_pass():
    """A second pass adds 5 us to an evaluation of 28, empty or not.  A call of the approximate solver, whose
    batches are counted where deferrals are, does not bring it.  Medians of 40 evaluations of each kind, in turn."""
    ctx = css.create(0)
    ico = synth.icosphere(3, 1.0)
    mesh = css.mesh_upload(ctx, ico.verts, ico.faces)
    parts = css.particles_set(ctx, mesh, *synth.place_uniform(ico, 60, 3))
    alone, after = [], []
    for _ in range(40):
        for us, solver in ((alone, False), (after, True)):
            assert _deferred(ctx, parts, 0.1) == 0
            if solver:
                css.vhm_neighbors(parts, 0.3, 1.0)
                assert ctx.last_counters()["deferred"] > 0
            assert _deferred(ctx, parts, 0.1) == 0
            us.append(1e3 * ctx.last_kernel_ms())
    parts.free()
    mesh.free()
    ctx.close()
    assert np.median(after) < np.median(alone) + 3.5, (np.median(after), np.median(alone))


def test_kernel_time_holds_no_round_trip():
    """The first evaluation of a set that defers sources launches the second pass once the host has seen them,
    later ones with the first: css_last_kernel_ms is the same device time, 870 us here, where the round
    trip between the passes takes 20 us."""
    ctx = css.create(0)
    ctx.set_launch(**dict(ctx.get_launch(), window_capacity=64))
    m = synth.icosphere(5, 1.0, noise=0.01, seed=1)
    face, bary = synth.place_uniform(m, 1024, 3)
    mesh = css.mesh_upload(ctx, m.verts, m.faces)
    other = css.particles_set(ctx, mesh, face[:2], bary[:2])
    late, once = [], []
    for _ in range(15):
        parts = css.particles_set(ctx, mesh, face, bary)
        assert _deferred(ctx, other, 1e-6) == 0
        for us in (late, once):
            assert _deferred(ctx, parts, 0.15) > 0
            us.append(1e3 * ctx.last_kernel_ms())
        parts.free()
    other.free()
    mesh.free()
    ctx.close()
    assert np.median(late) < np.median(once) + 10.0, (np.median(late), np.median(once))


def test_tuner_times_each_kernel_once():
    """Occupancy 1 and 2 are the same kernel: the tuner does not let noise choose between them."""
    m = synth.icosphere(4, 1.0, noise=0.01, seed=1)
    ctx = css.create(0)
    mesh = css.mesh_upload(ctx, m.verts, m.faces)
    parts = css.particles_set(ctx, mesh, *synth.place_uniform(m, 300, 3))
    pot = dict(kind=css.POT_HARMONIC, eps=1.0, sigma=0.2, r_cut=0.2, A=1.0)
    for _ in range(3):
        assert ctx.autotune([parts], pot, 0.2, css.FP64, reps=1)[0]["occupancy"] == 1
    parts.free()
    mesh.free()
    ctx.close()
