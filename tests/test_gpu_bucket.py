"""Bucketing and row starts in one CTA against the general launches: the rows of a set of n
particles equal the first n rows of the same set with particles added out of reach that
take it over the one-CTA forms' sizes (needs a GB300).

Distances of one pair may come from another launch shape, so they are compared to 1e-14 of
the distance (some tens of roundings of 1.1e-16 along the unfolding)."""
import numpy as np
import pytest

import synth

css = pytest.importorskip("paper_2404_19751_gb300")
pytestmark = pytest.mark.gpu


def _rows(ctx, mesh, face, bary, r_c):
    parts = css.particles_set(ctx, mesh, face, bary)
    out = css.geodesic_neighbors(parts, r_c, css.FP64)
    parts.free()
    return out


@pytest.mark.parametrize("n,general,crowded", [(1, 4097, 0), (2, 4097, 0), (40, 4097, 40), (511, 4097, 33),
                                               (2049, 4097, 32), (4096, 4097, 0), (8192, 8193, 0)])
def test_one_cta_forms_match_general(n, general, crowded):
    m = synth.icosphere(4, 1.0, noise=0.0, seed=2)
    c = np.asarray(m.verts)[np.asarray(m.faces)].mean(1)
    near, far = np.where(c[:, 2] > 0.2)[0], np.where(c[:, 2] < -0.2)[0]
    rng = np.random.default_rng(n)
    face = rng.choice(near, n).astype(np.int32)
    face[:crowded] = near[7]
    face = np.concatenate([face, rng.choice(far, general - n).astype(np.int32)])
    bary = rng.dirichlet((2.0, 2.0, 2.0), general)
    ctx = css.create(0)
    mesh = css.mesh_upload(ctx, m.verts, m.faces, m.period)
    r_c = min(0.3, 3.0 / np.sqrt(n))
    a = _rows(ctx, mesh, face[:n], bary[:n], r_c)
    b = _rows(ctx, mesh, face, bary, r_c)
    mesh.free()
    ctx.close()
    k = int(a[0][-1])
    assert np.array_equal(a[0], b[0][:n + 1])
    assert np.array_equal(a[1], b[1][:k])
    assert np.all(np.abs(a[2] - b[2][:k]) <= 1e-14 * np.maximum(a[2], 1e-3))
    if n >= 40:
        assert k > 0
