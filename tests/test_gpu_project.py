"""The projection's staged SH coefficients and view ranges where blocks and
16-byte pieces end unevenly: every degree and storage type, scenes of a few
Gaussians more or less than a block, one view and many."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,deg,dtype,views", [
    (1, 3, "f32", 1), (5, 2, "f16", 7), (255, 1, "bf16", 45), (256, 0, "f32", 3),
    (257, 3, "f16", 45), (257, 2, "bf16", 5), (513, 1, "f32", 37), (767, 0, "f16", 2),
    (1300, 3, "bf16", 61), (1300, 2, "f32", 11),
])
def test_projection_edges(n, deg, dtype, views):
    from paper_2407_14053_gb300 import Renderer
    scene = W.make_scene(W.SceneSpec(n, deg, "uniform", dtype, seed=n + deg))
    d = W.Display(67, 41, views, 5.3, 1 / 6, view_span_deg=12.0)
    r = Renderer(0)
    sid, did = r.load_gaussians(scene, dtype), r.set_display(d)
    L0 = W.light_field_centre(4.0, 1.0)
    V = oracle.view_map(d)
    ref = oracle.render_subpixels(oracle.Scene(W.quantise_storage(scene, dtype)), d, L0,
                                  np.arange(3 * d.width * d.height), V, oracle.repurpose(d, V))
    for where in ("two_pass", "projection"):
        r.set_key_emission(where)
        for _ in range(3):  # sized, laid out, emitted by the projection
            img = r.render(sid, did, L0, "directl").cpu().numpy().reshape(-1)
            assert r.stats()["status"] == 0
            assert ((img >= ref["lo"] - 2e-3) & (img <= ref["hi"] + 2e-3)).all()
    r.close()


@pytest.mark.parametrize("mode", ["directl", "raycast"])
@pytest.mark.parametrize("n,w,h,views", [(60, 24, 16, 3), (2000, 240, 135, 45), (40000, 320, 200, 9)])
def test_frames_back_to_back(mode, n, w, h, views):
    """A frame's kernels start while the ones before them drain: frames enqueued
    one behind the other, moving nearer and farther so that some emit their keys
    again, equal the same frames rendered with a wait after each."""
    from paper_2407_14053_gb300 import Renderer
    import torch
    scene = W.make_scene(W.SceneSpec(n, 1, "uniform", "f32", seed=n))
    d = W.Display(w, h, views, 5.3, 1 / 6, view_span_deg=12.0)
    poses = [W.light_field_centre(4.0 + 0.4 * (i % 5), 0.3 * i) for i in range(12)]
    frames = []
    for wait in (True, False):
        r = Renderer(0)
        sid, did = r.load_gaussians(scene, "f32"), r.set_display(d)
        for distance in (4.0, 4.0):
            r.render(sid, did, W.light_field_centre(distance, 0.0), mode)
        got = []
        for L0 in poses:
            got.append(r.render(sid, did, L0, mode).clone())
            if wait:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        frames.append([g.cpu().numpy() for g in got])
        r.close()
    for a, b in zip(*frames):
        assert np.array_equal(a, b)
    assert max(f.max() for f in frames[0]) > 0.05
