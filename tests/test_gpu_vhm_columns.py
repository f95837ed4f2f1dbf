"""The approximate solver's two forms against its FP64 oracle: one column per cluster where
a column fits in shared memory (cluster sizes 1, 2, 4 and 8 by the number of sources), and
the general form above that size.  Tolerances are those of the solver's other tests: 1e-9 of
the larger of the distance and the mesh spacing, 1e-7 for tangents (needs a GB300)."""
import math

import numpy as np
import pytest

import synth
from oracle import vhm as V

css = pytest.importorskip("paper_2404_19751_gb300")
pytestmark = pytest.mark.gpu


def _fan(k):
    """A closed double cone over a k-gon: two vertices of degree k, the others of degree 4."""
    a = 2 * math.pi * np.arange(k) / k
    v = np.concatenate([np.stack([np.cos(a), np.sin(a), 0 * a], 1), [[0.0, 0.0, 0.7], [0.0, 0.0, -0.7]]])
    f = [(i, (i + 1) % k, k) for i in range(k)] + [((i + 1) % k, i, k + 1) for i in range(k)]
    return synth.Mesh(v, np.array(f, np.int32), None)


CASES = {   # mesh, sources, time factor
    "two_sources": (lambda: synth.icosphere(3, 1.0, noise=0.02, seed=1), 2, 1.0),
    "cluster_8_odd_degrees": (lambda: _fan(37), 11, 1.0),
    "cluster_4": (lambda: synth.torus(2.0, 0.7, 31, 17), 30, 1.0),
    "cluster_2_boundary": (lambda: synth.holed_plane(21, (0.4, 0.6, 0.4, 0.6)), 70, 0.3),
    "cluster_1_periodic": (lambda: synth.periodic_heightfield(19, 6, seed=3), 153, 5.0),
    "largest_in_shared": (lambda: synth.torus(3.0, 1.0, 204, 68), 5, 1.0),
    "general": (lambda: synth.torus(3.0, 1.0, 210, 70), 5, 1.0),
}


@pytest.mark.parametrize("name", list(CASES))
def test_vhm_forms_match_oracle(name):
    make, n, tf = CASES[name]
    m = make()
    face, bary = synth.place_uniform(m, n, 17)
    om = V.VhmMesh(m, t_factor=tf)
    r = om.neighbors(face, bary, math.inf)
    ctx = css.create(0)
    mesh = css.mesh_upload(ctx, m.verts, m.faces, m.period)
    parts = css.particles_set(ctx, mesh, face, bary)
    a = css.vhm_neighbors(parts, math.inf, tf)
    b = css.vhm_neighbors(parts, math.inf, tf)
    parts.free()
    mesh.free()
    ctx.close()
    for x, y in zip(a, b):   # sums in a fixed order
        assert np.array_equal(x, y)
    assert np.array_equal(a[0], r[0]) and np.array_equal(a[1], r[1])
    assert np.max(np.abs(a[2] - r[2]) / np.maximum(np.abs(r[2]), om.h)) <= 1e-9
    assert np.max(np.linalg.norm(a[3] - r[3], axis=1)) <= 1e-7
