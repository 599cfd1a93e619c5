"""Kernel timers with enclosures that run in x_1 ranges (a level whose children would not fit
in one tree)."""
import numpy as np
import pytest

from paper_2406_09857_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k,degree,depth,cap", [(2, 6, 8, 200),    # small trees all the way
                                                (3, 8, 7, 60000)])  # and large ones
def test_timers_where_a_level_overflows(vx, k, degree, depth, cap):
    polys = [synth.kostlan_poly(k, degree, 8100 + k)]
    dom = synth.cube(k)
    s = vx.System(polys)
    plain = vx.enclose_system(s, dom, depth, vx.make_opts(vx.FP64))
    assert plain.stats()["tested"].max() > cap
    for mode in (vx.FP64, vx.FP32):
        o = vx.make_opts(mode, max_level_boxes=cap, timing=True)
        r = vx.enclose_system(s, dom, depth, o)
        assert np.array_equal(r.boxes(), plain.boxes())
        wall = r.elapsed_ms()
        for name, v in r.timing().items():
            assert 0.0 <= v["ms"] <= wall, (name, v, wall)
