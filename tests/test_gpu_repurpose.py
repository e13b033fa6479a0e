"""Repurposing (Alg. 2) by four lanes per (area, view), bit-exact against the
oracle where a view's subpixels sit differently in their units: several or
none a unit, units narrower than a subpixel or wider than the panel, areas
wider than the panel, windows that clip at every border."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [
    dict(width=90, height=50, num_views=2, pitch_lx=30.0, tan_slant=0.25),
    dict(width=50, height=70, num_views=300, pitch_lx=7.3, tan_slant=0.11, offset_k=-900.0),
    dict(width=40, height=30, num_views=9, pitch_lx=0.7, tan_slant=0.2, p_w=5),
    dict(width=61, height=40, num_views=20, pitch_lx=9.1, tan_slant=-2.3, p_w=1),
    dict(width=64, height=33, num_views=12, pitch_lx=4.5, tan_slant=1.9, p_w=2),
    dict(width=30, height=60, num_views=45, pitch_lx=1000.0, tan_slant=0.3, offset_k=500.0),
    dict(width=45, height=37, num_views=45, pitch_lx=5.3, tan_slant=1 / 6, p_w=2**31 - 1),
    dict(width=200, height=2, num_views=45, pitch_lx=5.3, tan_slant=1 / 6),
    dict(width=3, height=200, num_views=31, pitch_lx=6.25, tan_slant=0.0, offset_k=1e6),
])
def test_repurposing_edges(kw):
    from paper_2407_14053_gb300 import Renderer
    d = W.Display(**kw)
    r = Renderer(0)
    did = r.set_display(d)
    src = r.subpixel_map(did)
    assert np.array_equal(src, oracle.repurpose(d, oracle.view_map(d)))
    r.close()
