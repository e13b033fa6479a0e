"""Ray-order frames captured into the caller's graph: replays give the frame,
and so do the calls after the capture."""
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu

L0 = W.light_field_centre(4.0, 1.0)


def _capture(r, sid, did, out):
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g):
        r.render(sid, did, L0, "raycast", out)
    return g


@pytest.mark.parametrize("sized", [True, False])
def test_captured_ray_order_frames(sized):
    from paper_2407_14053_gb300 import Renderer
    d = W.Display(160, 90, 7, 5.3, 1 / 6, view_span_deg=10.0)
    r = Renderer(0)
    sid = r.load_gaussians(W.make_scene(W.SceneSpec(1500, 1, "uniform", "f32", seed=6)), "f32")
    first, did = r.set_display(d), r.set_display(d.replace(height=80))
    r.render(sid, first, L0, "raycast")  # builds what the scene keeps
    if sized:
        for _ in range(3):
            want = r.render(sid, did, L0, "raycast").clone()
    out = torch.zeros(80, 160, 3, device="cuda")
    g = _capture(r, sid, did, out)
    if not sized:
        want = r.render(sid, did, L0, "raycast").clone()
    assert want.max() > 0.05
    for yaw in (1.0, 2.0, 3.0, 4.0):
        other = r.render(sid, did, W.light_field_centre(4.0, yaw), "raycast").clone()
        out.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert (out - want).abs().max() < 1e-5  # (a frame captured unsized walks the tree)
        if sized:
            assert torch.equal(out, want)
        assert torch.equal(other, want) == (yaw == 1.0)
    r.stats()
    r.close()
