"""Empty-space skipping of the ray marcher on volumes whose level 2 is large: the
map of where climbs end is built level by level from its parents (odd extents,
rows of one voxel, several levels), and frames of few pixels on them.  Samples
per pixel as the oracle takes them; the image is that of the frame without
skipping, bit for bit."""
import numpy as np
import pytest

import oracle
from paper_2009_02702_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mg():
    from paper_2009_02702_gb300 import mg as _mg
    _mg.lib()
    return _mg


# level-2 voxels 99,846 and 656,250 and 68,750; above 65,536 a level has its own launch
@pytest.mark.parametrize("dims,shown", [((1030, 514, 10), 6), ((1500, 700, 40), 1), ((3, 1100, 1000), 12),
                                        ((1030, 514, 10), 0)])
def test_skipping_on_large_levels(mg, dims, shown):
    S = 40
    vol = synth.make_volume(1, dims=dims, S=S)
    g = mg.mg_build(torch.from_numpy(vol).cuda(), S)
    og = oracle.Graph(vol, S)
    tf = synth.make_tf(1, S, 4)
    tf[shown:, 3] = 0.0
    vals = mg.mg_propagate_tf(g, torch.from_numpy(tf).cuda())
    ref_vals = oracle.propagate(og.p, og.q, og.a, og.b, S, tf.astype(np.float64)).astype(np.float32)
    opac = vals[:, 3].contiguous()
    for size, kw in (((40, 24), dict(lod_bias=0, base_step=0.5)), ((1, 1), dict(lod_bias=-1, base_step=0.5)),
                     ((33, 17), dict(lod_bias=2, base_step=1.0))):
        cam = synth.orbit_camera(1, dims=dims, width=size[0], height=size[1], ert=2.0, **kw)
        img, steps = mg.mg_raymarch(g, vals, cam, steps=True)
        img_s, steps_s = mg.mg_raymarch(g, vals, cam, opacity=opac, steps=True)
        mg.mg_sync_status(g)
        assert torch.equal(img, img_s)
        assert bool((steps_s <= steps).all())
        _, ref_steps, _ = og.raymarch(ref_vals, cam, opacity=ref_vals[:, 3].copy())
        assert np.array_equal(steps_s.cpu().numpy(), ref_steps)
    g.close()


def test_values_that_are_not_finite(mg):
    """Samples inside one node take its value without the interpolation's seven
    steps: infinities and NaNs come out as they would."""
    dims, S = (48, 40, 36), 30
    vol = synth.make_volume(1, dims=dims, S=S)
    g = mg.mg_build(torch.from_numpy(vol).cuda(), S)
    og = oracle.Graph(vol, S)
    tf = synth.make_tf(1, S, 4)
    tf[3, 0], tf[7, 1], tf[11, 2] = np.inf, -np.inf, np.nan
    vals = mg.mg_propagate_tf(g, torch.from_numpy(tf).cuda())
    cam = synth.orbit_camera(1, dims=dims, width=96, height=64, lod_bias=0, ert=2.0, base_step=0.5)
    img = mg.mg_raymarch(g, vals, cam).cpu().numpy()
    ref, _, _ = og.raymarch(vals.cpu().numpy(), cam)
    assert np.isnan(ref).any()
    assert np.array_equal(np.isnan(img), np.isnan(ref)) and np.array_equal(np.isinf(img), np.isinf(ref))
    fin = np.isfinite(ref)
    assert np.abs(img[fin] - ref[fin]).max() <= 2e-5
    mg.mg_sync_status(g)
    g.close()


def test_extents_that_an_image_only_claims(mg):
    """An imported image may give a level's extents in another order: climbs stay
    inside the levels' arrays, as the samples do."""
    dims, S = (64, 64, 8), 12
    g = mg.mg_build(torch.from_numpy(synth.make_volume(1, dims=dims, S=S)).cuda(), S)
    img = np.array(mg.mg_graph_export(g))
    at = 64   # the header's extents, three int32 a level
    ext = img[at:at + 12 * g.info["levels"]].view(np.int32).reshape(-1, 3)
    assert ext.tolist() == [list(d) for d in g.info["dims"]] and ext[2].tolist() == [16, 16, 2]
    ext[2] = (2, 16, 16)
    h = mg.mg_graph_import(img)
    vals = mg.mg_propagate_tf(h, torch.from_numpy(synth.make_tf(1, S, 4)).cuda())
    cam = synth.orbit_camera(1, dims=dims, width=33, height=17, lod_bias=0, ert=2.0, base_step=0.5)
    out = mg.mg_raymarch(h, vals, cam, opacity=torch.zeros(h.N, device="cuda"))
    mg.mg_sync_status(h)
    assert bool(torch.isfinite(out).all())
    g.close()
    h.close()
