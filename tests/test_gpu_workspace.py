"""The neighbour kernel's workspace: bounded by the work and by the device's free memory, with the same
rows whatever it gets (needs a GB300).  A capacity of 2^20 windows makes a slice 68 MB, as the shapes
picked for large patches do; the patches here are small, so the calls are short."""
import numpy as np
import pytest

import synth

css = pytest.importorskip("paper_2404_19751_gb300")
torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPE = dict(warps_per_cta=4, ctas_per_sm=0, tile=1, shared_scale=0, window_capacity=1 << 20,
             window_capacity2=16384, warps2_per_sm=2, occupancy=1, table_capacity=0, team=0)


def _call(ctx, m, face, bary, r_c):
    mesh = css.mesh_upload(ctx, m.verts, m.faces, m.period)
    parts = css.particles_set(ctx, mesh, face, bary)
    before = torch.cuda.mem_get_info()[0]
    g = css.geodesic_neighbors(parts, r_c, css.FP64)
    taken = before - torch.cuda.mem_get_info()[0]
    parts.free()
    mesh.free()
    return g, taken


@pytest.mark.parametrize("team", [0, 1])
def test_little_free_memory_gives_the_same_rows(team):
    """Slices for 400 groups or teams would take 27 GB; with 3 GB left fewer of them run, on the first call and
    on later ones."""
    m = synth.icosphere(3, 1.0, noise=0.03, seed=3)
    face, bary = synth.place_uniform(m, 400, 4)
    got = []
    for left in (None, 3 << 30):
        torch.cuda.empty_cache()
        hold = None
        if left:
            hold = torch.empty(torch.cuda.mem_get_info()[0] - left, dtype=torch.uint8, device="cuda")
        ctx = css.create(0)
        if left:
            ctx.set_launch(**dict(SHAPE, team=team))
        for _ in range(2):
            got.append(_call(ctx, m, face, bary, 0.5)[0])
        ctx.close()
        del hold
    torch.cuda.empty_cache()
    assert len(got[0][1]) > 1000
    for g in got[1:]:
        assert np.array_equal(got[0][0], g[0]) and np.array_equal(got[0][1], g[1])
        np.testing.assert_allclose(g[2], got[0][2], rtol=1e-13, atol=0)


def test_few_sources_take_few_slices():
    """64 sources take a slice each, not one for each of the 304 teams that could be resident (20 GB)."""
    m = synth.icosphere(3, 1.0, noise=0.03, seed=3)
    face, bary = synth.place_uniform(m, 64, 4)
    ctx = css.create(0)
    ctx.set_launch(**dict(SHAPE, team=1, warps_per_cta=8))
    _, taken = _call(ctx, m, face, bary, 0.5)
    ctx.close()
    assert taken < 6 << 30, taken
