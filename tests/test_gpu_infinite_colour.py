"""A Gaussian whose colour overflows to infinity colours the pixels that it
reaches and no others: the standard paradigm's kernels, by direct and by
transposed evaluation, on lists of every class."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,spread", [(60, 1.0), (1500, 0.6), (5000, 0.25)])
def test_an_infinite_colour_stays_where_it_is(n, spread):
    from paper_2407_14053_gb300 import Renderer
    scene = W.make_scene(W.SceneSpec(n, 0, "uniform", "f32", seed=n))
    scene["mean"] *= np.float32(spread)
    wild = np.arange(0, n, max(n // 3, 1))[:3]
    scene["sh"][wild, 0, 0] = np.inf
    scene["log_scale"][wild] = np.float32(-4.0)
    scene["opacity_logit"][wild] = np.float32(2.0)
    d = W.Display(64, 48, 3, 5.3, 1 / 6, view_span_deg=8.0)
    r = Renderer(0)
    sid, did = r.load_gaussians(scene, "f32"), r.set_display(d)
    L0 = W.light_field_centre(4.0, 1.0)
    direct = r.render(sid, did, L0, "standard").cpu().numpy()
    r.set_eval("standard", "transposed")
    transposed = r.render(sid, did, L0, "standard").cpu().numpy()
    assert np.array_equal(direct, transposed, equal_nan=True)
    # (among 5,000 the three lie behind opaque ones)
    assert np.isinf(direct).any() or n == 5000
    assert np.isfinite(direct).mean() > 0.8
    assert np.isfinite(direct[..., 1:]).all()  # the colour is infinite in red alone
    r.close()
