"""Repurposing (Alg. 2) on panels of a small pitch, bit-exact against the
oracle: pitches below a subpixel (units that no subpixel falls in, views that no
subpixel shows, areas narrower than a subpixel) and pitches that repeat after a
few subpixels, where few of the views are shown; and the time of the former."""
import time

import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [
    dict(width=60, height=40, num_views=12, pitch_lx=0.99, tan_slant=0.2),
    dict(width=60, height=40, num_views=45, pitch_lx=0.31, tan_slant=-0.25, p_w=3),
    dict(width=50, height=44, num_views=7, pitch_lx=0.5, tan_slant=0.0, p_w=1, offset_k=-3.3),
    dict(width=90, height=33, num_views=20, pitch_lx=0.013, tan_slant=0.17),
    dict(width=90, height=33, num_views=20, pitch_lx=0.013, tan_slant=-0.17, p_w=500),
    dict(width=41, height=37, num_views=300, pitch_lx=0.07, tan_slant=1.3, offset_k=900.0),
    dict(width=45, height=37, num_views=9, pitch_lx=0.25, tan_slant=0.5, p_w=2**31 - 1),
    dict(width=1, height=5, num_views=3, pitch_lx=0.4, tan_slant=-1.1),
    # few views shown, and just not few
    dict(width=70, height=50, num_views=45, pitch_lx=1.5, tan_slant=1 / 6),
    dict(width=70, height=50, num_views=45, pitch_lx=2.0, tan_slant=0.0, offset_k=0.25, p_w=3),
    dict(width=70, height=50, num_views=45, pitch_lx=3.0, tan_slant=-1 / 6, p_w=1),
    dict(width=70, height=50, num_views=100, pitch_lx=3.4, tan_slant=1 / 3, p_w=2**31 - 1),
    dict(width=70, height=50, num_views=12, pitch_lx=3.4, tan_slant=0.171),
    dict(width=70, height=50, num_views=65535, pitch_lx=1.37, tan_slant=0.171),
])
def test_repurposing_at_a_small_pitch(kw):
    from paper_2407_14053_gb300 import Renderer
    d = W.Display(**kw)
    r = Renderer(0)
    did = r.set_display(d)
    assert np.array_equal(r.view_map(did), oracle.view_map(d))
    assert np.array_equal(r.subpixel_map(did), oracle.repurpose(d, oracle.view_map(d)))
    r.close()


@pytest.mark.parametrize("tan", [0.1646, -0.1646])
def test_a_small_pitch_takes_no_longer_by_its_units(tan):
    """A window of the search holds at most a row's subpixels, however many
    units fall in it: 30 times the set-up of a panel of the same size at pitch
    5.4 is ample for one at 0.01 (looking at every unit took 70 to 600 times)."""
    import torch
    from paper_2407_14053_gb300 import Renderer
    r = Renderer(0)

    def set_up(pitch):
        best = 1e9
        for _ in range(3):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            did = r.set_display(W.Display(480, 270, 45, pitch, tan, view_span_deg=10.0))
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - t0)
            r.free_display(did)
        return best

    assert set_up(0.0101379) < 30 * set_up(5.373)
    r.close()
