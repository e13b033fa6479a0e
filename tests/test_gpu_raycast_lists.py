"""Ray-order frames from tile lists: the lists must hold every Gaussian that a
ray meets, whatever its outline, and a frame whose lists do not fit walks the
tree."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def renderer():
    from paper_2407_14053_gb300 import Renderer
    r = Renderer(0)
    yield r
    r.close()


def _check(img, scene, d, L0, sub, cap=128):
    V = oracle.view_map(d)
    ref = oracle.raycast_subpixels(oracle.Scene(scene), d, L0, sub, V, oracle.repurpose(d, V), cap)
    got = img.reshape(-1)[sub]
    assert ((got >= ref["lo"] - 2e-3) & (got <= ref["hi"] + 2e-3)).all()


# thin and long (up to 55 : 1; from about 400 : 1 on the exact test's FP32
# rounding itself passes 2e-3, on the tree as on the lists), huge (whole views), around and behind the cameras, sub-pixel;
# lists of several sorted chunks; heaps that overflow; groups of over 32 rays
@pytest.mark.parametrize("n,scale,aspect,spread,distance,cap,views,rig", [
    (400, -2.5, 3.0, 1.0, 4.0, 128, 12, 0),
    (300, -3.0, 4.0, 1.0, 4.0, 256, 5, 1),
    (200, 0.0, 0.5, 1.0, 2.0, 128, 3, 0),
    (500, -2.0, 0.5, 2.0, 0.5, 128, 4, 0),
    (3000, -7.0, 0.5, 1.0, 4.0, 16, 6, 0),
    (2500, -2.5, 0.5, 0.15, 4.0, 64, 2, 0),
    (1, -1.0, 0.0, 0.1, 4.0, 1, 1, 0),
])
def test_lists_match_the_oracle(renderer, n, scale, aspect, spread, distance, cap, views, rig):
    r = renderer
    scene = W.make_scene(W.SceneSpec(n, 2, "uniform", "f32", seed=n))
    scene["mean"] *= np.float32(spread)
    scene["log_scale"][:] = np.float32(scale)
    scene["log_scale"][:, 0] -= np.float32(aspect)
    d = W.Display(70, 45, views, 5.3, 1 / 6, view_span_deg=15.0, rig=rig)
    sid, did = r.load_gaussians(scene, "f32"), r.set_display(d)
    r.set_heap_capacity(cap)
    try:
        for yaw in (0.0, 3.0):  # sized, then laid out by the frame before
            L0 = W.light_field_centre(distance, yaw)
            img = r.render(sid, did, L0, "raycast").cpu().numpy()
            _check(img, scene, d, L0, np.arange(img.size), cap)
    finally:
        r.set_heap_capacity(128)
        r.free_display(did)
        r.free_scene(sid)


def test_a_frame_that_outgrows_its_lists_is_complete(renderer):
    """Far away every Gaussian is in a tile or two; from among them each one
    fills the view, many times the keys that were sized for."""
    r = renderer
    scene = W.make_scene(W.SceneSpec(2000, 1, "uniform", "f32", seed=2))
    scene["mean"] *= np.float32(0.3)
    d = W.Display(320, 200, 4, 5.3, 1 / 6, view_span_deg=10.0)
    sid, did = r.load_gaussians(scene, "f32"), r.set_display(d)
    sub = W.sample_subpixels(d, 200, windows=1, window_px=6, seed=1)
    for distance in (60.0, 0.3, 0.3, 60.0):
        L0 = W.light_field_centre(distance, 1.0)
        img = r.render(sid, did, L0, "raycast").cpu().numpy()
        _check(img, scene, d, L0, sub)
    r.free_display(did)
    r.free_scene(sid)


# four lanes blend a ray where the SH coefficients are whole 16-byte pieces (3,
# 6 or 12 of them), one lane where they are not; lists shorter than four, not a
# multiple of four, and cut by the transmittance
@pytest.mark.parametrize("dtype,degree", [("f32", 0), ("f32", 1), ("f32", 3), ("bf16", 1),
                                          ("bf16", 3), ("f16", 3)])
@pytest.mark.parametrize("cap", [1, 6, 128])
def test_blending_by_pieces(renderer, dtype, degree, cap):
    r = renderer
    scene = W.make_scene(W.SceneSpec(900, degree, "uniform", dtype, seed=degree + cap))
    d = W.Display(37, 29, 5, 5.3, 1 / 6, view_span_deg=15.0)
    sid, did = r.load_gaussians(scene, dtype), r.set_display(d)
    r.set_heap_capacity(cap)
    try:
        L0 = W.light_field_centre(3.0, 1.0)
        img = r.render(sid, did, L0, "raycast").cpu().numpy()
        stored = scene if dtype == "f32" else W.quantise_storage(scene, dtype)
        _check(img, stored, d, L0, np.arange(img.size), cap)
    finally:
        r.set_heap_capacity(128)
        r.free_display(did)
        r.free_scene(sid)
