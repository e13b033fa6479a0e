"""What a ray-order frame reports of its lists, and with that: frames whose
keys outgrow their slices are emitted again, frames that outgrow the key buffer
walk the tree, and both are the frames of lists that fit."""
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


def test_ray_order_frames_report_their_lists():
    from paper_2407_14053_gb300 import Renderer
    scene = W.make_scene(W.SceneSpec(3000, 1, "uniform", "f32", seed=8))
    scene["mean"] *= 0.3
    d = W.Display(200, 120, 4, 5.3, 1 / 6, view_span_deg=10.0)
    r = Renderer(0)
    sid, did = r.load_gaussians(scene, "f32"), r.set_display(d)

    def frame(distance, yaw=0.0):
        out = r.render(sid, did, W.light_field_centre(distance, yaw), "raycast").clone()
        return out, r.stats()

    far, st = frame(30.0)
    lists = st["lists_small"]
    assert lists > 0 and st["n_keys"] >= 3000 and st["reemitted"] == 0 and st["status"] == 0
    _, st = frame(24.0, 1.0)  # other tiles than the frame before
    assert st["reemitted"] == 1 and st["lists_small"] == lists
    walked, st = frame(0.8)  # many times the keys
    assert st["reemitted"] == 1 and st["lists_small"] == 0
    near, st = frame(0.8)  # sized again
    assert st["reemitted"] == 0 and st["lists_small"] == lists
    # the same hits in the same order, summed in another
    assert (walked - near).abs().max() < 1e-5 and near.max() > 0.05
    again, st = frame(30.0)
    assert st["lists_small"] == lists and torch.equal(again, far)
    r.close()
