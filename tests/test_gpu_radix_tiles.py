"""The radix path at the largest standard tiles (1024 pixels, a block of 1024
threads): the frames of the binned path, bit for bit."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile", [(32, 32), (64, 16), (8, 128), (128, 8), (16, 32)])
def test_radix_at_the_largest_standard_tiles(tile):
    from paper_2407_14053_gb300 import Renderer
    scene = W.make_scene(W.SceneSpec(700, 1, "uniform", "f32", seed=3))
    d = W.Display(75, 41, 3, 5.3, 1 / 6, view_span_deg=8.0)
    r = Renderer(0)
    sid, did = r.load_gaussians(scene, "f32"), r.set_display(d)
    r.set_tile("standard", *tile)
    L0 = W.light_field_centre(4.0, 1.0)
    binned = r.render(sid, did, L0, "standard").cpu().numpy()
    r.set_sort_mode("radix")
    radix = r.render(sid, did, L0, "standard").cpu().numpy()
    assert np.array_equal(binned, radix)
    assert binned.max() > 0.05
    r.close()
