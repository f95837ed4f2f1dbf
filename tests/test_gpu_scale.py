"""The same surface in other units of length (needs a GB300).  Scaled by a power of two, every length
the library computes scales exactly, so distances and forces are the same bits times that power,
directions the same bits."""
import math

import numpy as np
import pytest

import synth

css = pytest.importorskip("paper_2404_19751_gb300")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = css.create(0)
    yield c
    c.close()


def _particles(m, n):
    face, bary = synth.place_uniform(m, n, 5)
    for k, eps in enumerate((1e-14, 1e-11, 1e-8, 1e-5)):   # next to a vertex
        bary[k] = np.roll([1.0 - 1.7 * eps, eps, 0.7 * eps], k)
    return face, bary


def _results(ctx, m, face, bary, scale, r_c, prec):
    mesh = css.mesh_upload(ctx, m.verts * scale, m.faces, None if m.period is None else tuple(p * scale for p in m.period))
    parts = css.particles_set(ctx, mesh, face, bary)
    pot = dict(kind=css.POT_WCA, eps=1.0, sigma=0.3 * scale, r_cut=0.3 * 2 ** (1 / 6) * scale, A=1.0)
    try:
        rows = css.geodesic_neighbors(parts, r_c * scale, prec)
        return rows, css.compute_forces(parts, pot, pot["r_cut"], prec)[0]
    finally:
        parts.free()
        mesh.free()


@pytest.mark.parametrize("power", [70, 200, -30, -70, -200])
@pytest.mark.parametrize("name,r_c", [("rough", 0.5), ("rough", math.inf), ("hfield", 0.3)])
def test_results_scale_exactly(ctx, name, r_c, power):
    m = {"rough": synth.icosphere(3, 1.0, noise=0.03, seed=2), "hfield": synth.periodic_heightfield(20, 8, seed=4)}[name]
    face, bary = _particles(m, 120)
    for prec in (css.FP64, css.FP32):
        a, fa = _results(ctx, m, face, bary, 1.0, r_c, prec)
        b, fb = _results(ctx, m, face, bary, 2.0 ** power, r_c, prec)
        assert len(a[1]) > 100
        assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
        assert np.array_equal(a[2] * 2.0 ** power, b[2])
        assert np.array_equal(a[3], b[3])
        assert np.array_equal(fa, fb * 2.0 ** power)
