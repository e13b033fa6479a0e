"""The standard paradigm's compositing kernels (a warp per tile list of up to
512 or 1024 keys, a block per longer list; 8 x 8 patches, two pixels a lane)
at the edges of their tiles, patches, runs and sorts."""
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


def _render(r, sid, did, L0, strategy=None, sort=None):
    try:
        if strategy:
            r.set_eval("standard", strategy)
        if sort:
            r.set_sort_mode(sort)
        out = r.render(sid, did, L0, "standard").cpu().numpy()
        return out, r.stats()
    finally:
        r.set_eval("standard", "direct")
        r.set_sort_mode("auto")


# Every path blends with the same operations in the same order, so frames are
# compared bit for bit; the oracle bounds them all at the FP32 tolerance.
@pytest.mark.parametrize("w,h,tile,n,spread,flat", [
    (1, 1, (16, 16), 40, 1.0, False),       # one pixel
    (7, 9, (8, 8), 300, 1.0, False),        # one patch and a row and column of the next
    (17, 33, (8, 32), 500, 1.0, False),     # quads that a tile fills by half
    (33, 15, (64, 16), 31, 1.0, False),     # fewer records than a batch
    (48, 40, (32, 32), 1000, 0.6, False),   # four quads a tile; lists around 512 and 1024
    (40, 40, (16, 16), 5000, 0.25, False),  # long lists: the block class
    (40, 40, (16, 16), 400, 0.3, True),     # equal depths: bitonic sort of a warp's list
    (40, 40, (32, 16), 3001, 0.25, True),   # and of a block's, not a power of two
])
def test_views_match_every_other_path_and_the_oracle(renderer, w, h, tile, n, spread, flat):
    r = renderer
    scene = W.make_scene(W.SceneSpec(n, 1, "uniform", "f32", seed=n))
    scene["mean"] *= np.float32(spread)
    scene["log_scale"] -= np.float32(0.5)
    d = W.Display(w, h, 3, 5.3, 1 / 6, view_span_deg=8.0, rig=1 if flat else 0)
    if flat:  # one plane parallel to every view: all depths equal
        scene["mean"][:, 2] = 0.0
        scene["opacity_logit"] -= np.float32(3.0)
    sid, did = r.load_gaussians(scene, "f32"), r.set_display(d)
    L0 = W.light_field_centre(4.0, 0.0)
    r.set_tile("standard", *tile)
    try:
        img, st = _render(r, sid, did, L0)
        if n == 5000 or n == 3001:
            assert st["max_list"] > 1024 and st["lists_large"] > 0
        other, _ = _render(r, sid, did, L0, strategy="transposed")
        assert np.array_equal(img, other)
        if tile[0] * tile[1] < 1024:  # the radix path's blocks of 1024 threads do not launch
            radix, _ = _render(r, sid, did, L0, sort="radix")
            assert np.array_equal(img, radix)
        if not flat:  # every order of equal depths is valid
            V = oracle.view_map(d)
            ref = oracle.render_subpixels(oracle.Scene(scene), d, L0, np.arange(img.size), V, None)
            got = img.reshape(-1)
            assert ((got >= ref["lo"] - 2e-3) & (got <= ref["hi"] + 2e-3)).all()
    finally:
        r.set_tile("standard", 16, 16)
        r.free_display(did)
        r.free_scene(sid)


def test_views_saturating_pixels_stop(renderer):
    """Opaque layers: every pixel reaches the transmittance stop inside a run
    of records, at a different one."""
    r = renderer
    scene = W.make_scene(W.SceneSpec(900, 0, "uniform", "f32", seed=4))
    scene["opacity_logit"][:] = np.float32(3.0)
    scene["log_scale"][:] = np.float32(-1.5)
    d = W.Display(50, 30, 4, 5.3, 1 / 6, view_span_deg=8.0)
    sid, did = r.load_gaussians(scene, "f32"), r.set_display(d)
    L0 = W.light_field_centre(4.0, 2.0)
    img, _ = _render(r, sid, did, L0)
    other, _ = _render(r, sid, did, L0, strategy="transposed")
    assert np.array_equal(img, other)
    ref = oracle.render_subpixels(oracle.Scene(scene), d, L0, np.arange(img.size),
                                  oracle.view_map(d), None)
    got = img.reshape(-1)
    assert ((got >= ref["lo"] - 2e-3) & (got <= ref["hi"] + 2e-3)).all()
    r.free_display(did)
    r.free_scene(sid)


def test_views_keys_outgrow_their_slices(renderer):
    """The projection emits a frame's keys into slices laid out from the frame
    before: a small move fits, a larger one emits again, and one that needs
    many times the keys is rendered again from the start.  Every frame is the
    radix path's."""
    r = renderer
    scene = W.make_scene(W.SceneSpec(3000, 1, "uniform", "f32", seed=8))
    scene["mean"] *= np.float32(0.3)
    d = W.Display(200, 120, 4, 5.3, 1 / 6, view_span_deg=10.0)
    sid, did = r.load_gaussians(scene, "f32"), r.set_display(d)
    poses = [(30.0, 0.0), (30.0, 0.2), (24.0, 1.0), (0.8, 0.0), (0.8, 0.1), (30.0, 0.0)]
    L0s = [W.light_field_centre(distance, yaw) for distance, yaw in poses]
    frames = [_render(r, sid, did, L0) for L0 in L0s]
    for L0, (img, st) in zip(L0s, frames):
        radix, _ = _render(r, sid, did, L0, sort="radix")
        assert np.array_equal(img, radix)
    assert any(st["reemitted"] for _, st in frames)
    r.free_display(did)
    r.free_scene(sid)
