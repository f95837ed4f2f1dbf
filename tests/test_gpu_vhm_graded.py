"""The approximate solver on a mesh whose edges grow tenfold along both axes: the result is the
oracle's, and the over-relaxed sweeps are fewer than plain Gauss-Seidel sweeps would be (needs a
GB300)."""
import math

import numpy as np
import pytest
import scipy.sparse as sp
import scipy.sparse.linalg as spla

import synth
from oracle import vhm as V

css = pytest.importorskip("paper_2404_19751_gb300")
pytestmark = pytest.mark.gpu


def _graded(n, ratio):
    """The unit square on n x n vertices, spacings growing geometrically from 1 to ratio."""
    x = np.concatenate([[0.0], np.cumsum(ratio ** (np.arange(n - 1) / (n - 2.0)))])
    m = synth.grid_plane(n, n)
    k = np.arange(n * n)
    v = np.stack([x[k % n], x[k // n], 0.0 * k], 1)
    v[:, :2] /= x[-1]
    return synth.Mesh(v, m.faces, None)


def _plain_sweeps(A, b):
    """Gauss-Seidel sweeps from zero until the last of eight changes no entry by more than 1e-14 of
    the terms it is summed from."""
    low = spla.splu(sp.tril(A).tocsc(), permc_spec="NATURAL", diag_pivot_thresh=0.0)
    up, D = sp.triu(A, 1).tocsr(), A.diagonal()
    off = abs(A - sp.diags(D))
    x = np.zeros(len(b))
    for sweep in range(1, 5000):
        y = low.solve(b - up @ x)
        if sweep % 8 == 0 and not (np.abs(y - x) > 1e-14 * (off @ np.abs(y) + b) / D).any():
            return sweep
        x = y
    return sweep


@pytest.mark.parametrize("ratio", [4.0, 10.0])
def test_graded_mesh(ratio):
    m = _graded(64, ratio)
    face, bary = synth.place_uniform(m, 24, 7)
    face[0], bary[0] = m.nf - 1, [0.05, 0.05, 0.9]   # in the coarse corner
    face[1], bary[1] = 0, [0.9, 0.05, 0.05]          # in the fine one
    om = V.VhmMesh(m, t_factor=1.0)
    r = om.neighbors(face, bary, math.inf)
    ctx = css.create(0)
    mesh = css.mesh_upload(ctx, m.verts, m.faces, m.period)
    parts = css.particles_set(ctx, mesh, face, bary)
    g = css.vhm_neighbors(parts, math.inf, 1.0)
    sweeps = ctx.last_counters()["windows"]
    parts.free()
    mesh.free()
    ctx.close()
    assert np.array_equal(g[0], r[0]) and np.array_equal(g[1], r[1])
    # the bars of the solver's other tests
    assert np.max(np.abs(g[2] - r[2]) / np.maximum(np.abs(r[2]), om.h)) <= 1e-9
    assert np.max(np.linalg.norm(g[3] - r[3], axis=1)) <= 1e-7
    b = np.zeros(m.nv)
    b[-1] = 1.0
    plain = _plain_sweeps(sp.csr_matrix(om.M + om.t * om.L), b)
    assert sweeps < plain, (sweeps, plain)
