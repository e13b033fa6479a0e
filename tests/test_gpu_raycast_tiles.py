"""Ray-order frames from the lists of other tile shapes than the default: the
same hits, so the default's frame bit for bit, and the oracle's colours.  The
outline test expands an outline about its warp's rays, which lie up to 360
pixels apart in the largest tile; thin outlines of 30 to 70 pixels are where
its terms are largest."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale,aspect", [(-2.0, 4.0), (-1.4, 2.5), (-4.5, 0.5)])
def test_lists_of_any_tile_find_the_same_hits(scale, aspect):
    from paper_2407_14053_gb300 import Renderer
    scene = W.make_scene(W.SceneSpec(500, 1, "uniform", "f32", seed=int(-10 * scale)))
    scene["log_scale"][:] = np.float32(scale)
    scene["log_scale"][:, 0] -= np.float32(aspect)
    scene["log_scale"][:, 1] -= np.float32(aspect)
    d = W.Display(530, 260, 3, 5.3, 1 / 6, view_span_deg=8.0)
    L0 = W.light_field_centre(4.0, 1.0)
    r = Renderer(0)
    sid, did = r.load_gaussians(scene, "f32"), r.set_display(d)
    frame = r.render(sid, did, L0, "raycast").cpu().numpy()
    V = oracle.view_map(d)
    sub = W.sample_subpixels(d, 3000, windows=2, window_px=6, seed=1)
    ref = oracle.raycast_subpixels(oracle.Scene(scene), d, L0, sub, V, oracle.repurpose(d, V), 128)
    got = frame.reshape(-1)[sub]
    assert ((got >= ref["lo"] - 2e-3) & (got <= ref["hi"] + 2e-3)).all() and got.max() > 0.05
    for tile in ((8, 8), (128, 128), (256, 256), (256, 8)):
        r.set_tile("directl", *tile)
        for _ in range(2):  # sized, then laid out by the frame before
            assert np.array_equal(r.render(sid, did, L0, "raycast").cpu().numpy(), frame)
    r.close()
