"""Frames where device memory runs short: what a call cannot have costs that
call, and no other its frame."""
import numpy as np
import pytest
import torch

import workloads as W
from memory_pressure import free_bytes

pytestmark = pytest.mark.gpu

MB = 1 << 20


def _covering_scene(n, views_filled, seed=1):
    """n faint Gaussians; with views_filled each of them reaches every tile."""
    scene = W.make_scene(W.SceneSpec(n, 0, "uniform", "f32", seed=seed))
    if views_filled:
        scene["mean"] *= np.float32(0.1)
        scene["log_scale"][:] = np.float32(1.0)
        scene["opacity_logit"][:] = np.float32(-4.0)
    return scene


PANEL = W.Display(960, 540, 8, 5.3, 1 / 6, view_span_deg=8.0)
L0 = W.light_field_centre(4.0, 1.0)


@pytest.mark.parametrize("mode", ["directl", "standard"])
def test_a_key_buffer_that_cannot_grow_costs_no_other_frame(mode):
    """The key buffer is given up for a larger one that cannot be had: the
    frames of a signature sized before come out whole."""
    from paper_2407_14053_gb300 import DirectLError, Renderer
    r = Renderer(0)
    did = r.set_display(PANEL)
    small = r.load_gaussians(_covering_scene(400, False), "f32")
    large = r.load_gaussians(_covering_scene(4000, True), "f32")  # 4000 x 8 views x 510 tiles: 16 M keys
    want = r.render(small, did, L0, mode).clone()
    for _ in range(2):
        assert torch.equal(r.render(small, did, L0, mode), want)
    with free_bytes(96 * MB):  # of at least 130 for the keys alone
        with pytest.raises(DirectLError, match="OOM"):
            r.render(large, did, L0, mode)
        for _ in range(2):
            out = torch.full_like(want, -1.0)
            assert torch.equal(r.render(small, did, L0, mode, out), want)
    out = r.render(large, did, L0, mode)
    assert torch.isfinite(out).all() and out.max() > 0.05
    r.close()


def test_a_standard_frame_asks_for_its_views_first():
    """Room for M_m and the frame's keys (56 and 147 MB with the buffers'
    slack), but not for the larger key buffer (239 MB) of later frames as well."""
    from paper_2407_14053_gb300 import Renderer
    r = Renderer(0)
    did = r.set_display(PANEL)
    sid = r.load_gaussians(_covering_scene(1000, True), "f32")
    with free_bytes(250 * MB):
        first = r.render(sid, did, L0, "standard").clone()
        assert r.stats()["n_keys"] == 1000 * 8 * 60 * 34
        again = r.render(sid, did, L0, "standard").clone()
    assert torch.equal(first, again) and first.max() > 0.05
    later = [r.render(sid, did, L0, "standard").clone() for _ in range(70)]
    assert all(torch.equal(x, first) for x in later)
    r.close()


def test_what_is_kept_for_later_frames_is_given_back():
    """The ray-order renderer's intersection lists (900 MB here) do not keep a
    frame or a scene from the memory that it cannot do without, and are there
    again when the next ray-order frame wants them."""
    from paper_2407_14053_gb300 import Renderer
    r = Renderer(0)
    did = r.set_display(PANEL)
    sid = r.load_gaussians(_covering_scene(1000, True), "f32")
    rays = [r.render(sid, did, L0, "raycast").clone() for _ in range(2)]
    with free_bytes(64 * MB):
        standard = r.render(sid, did, L0, "standard").clone()  # 203 MB
    with free_bytes(64 * MB):
        directl = r.render(sid, did, L0, "directl").clone()
    rays.append(r.render(sid, did, L0, "raycast").clone())
    with free_bytes(64 * MB):
        other = r.load_gaussians(_covering_scene(600_000, False), "f32")  # 150 MB with its copies
    rays.append(r.render(sid, did, L0, "raycast").clone())
    assert all(torch.equal(x, rays[0]) for x in rays) and rays[0].max() > 0.05
    assert torch.equal(r.render(sid, did, L0, "standard"), standard)
    assert torch.equal(r.render(sid, did, L0, "directl"), directl)
    r.free_scene(other)
    r.close()


def _lists(r):  # a ray-order frame from tile lists is nine launches, a tree walk three
    return r.stats()["n_launches"] > 5


def test_ray_order_lists_are_asked_for_again():
    """Without memory for its lists (900 MB) a ray-order frame walks the tree;
    with less to ask for, or the memory free again, it has lists again."""
    from paper_2407_14053_gb300 import Renderer
    r = Renderer(0)
    warm = r.set_display(W.WORKLOADS["tiny"].display)
    did = r.set_display(PANEL)
    sid = r.load_gaussians(_covering_scene(1000, True), "f32")
    r.render(sid, warm, L0, "raycast")
    with free_bytes(400 * MB):
        walked = r.render(sid, did, L0, "raycast").clone()
        assert not _lists(r)
        assert torch.equal(r.render(sid, did, L0, "raycast"), walked) and not _lists(r)
        r.set_heap_capacity(16)  # 112 MB
        r.render(sid, did, L0, "raycast")
        assert _lists(r)
        r.set_heap_capacity(128)
        r.render(sid, did, L0, "raycast")
        assert not _lists(r)
    for _ in range(65):
        got = r.render(sid, did, L0, "raycast")
    assert _lists(r)
    assert (got - walked).abs().max() < 1e-5  # the same hits, blended in another order of sums
    r.close()


@pytest.mark.parametrize("heap", [16, 128])
def test_footprint_estimate_counts_the_intersection_lists(heap):
    from paper_2407_14053_gb300 import Renderer
    r = Renderer(0)
    did = r.set_display(PANEL)
    sid = r.load_gaussians(_covering_scene(20_000, False), "f32")
    r.set_heap_capacity(heap)
    lists = 8 * heap * r.display_info(did)[0]
    assert r.footprint(sid, did, "raycast") > lists > r.footprint(sid, did, "directl")
    r.close()
