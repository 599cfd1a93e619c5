"""Kernel timers with enclosures that run in x_1 ranges (a level whose children would not fit
in one tree), and the bytes that a small tree's prune is charged with."""
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


@pytest.mark.parametrize("k,depth", [(1, 9), (2, 6), (3, 4)])
def test_small_prunes_are_charged_their_own_bytes(vx, k, depth):
    """A keep byte per leaf, and 4 bytes per label, parent and first-child index of the nodes
    read and of the nodes written."""
    s = vx.System([synth.kostlan_poly(k, 5, 8200 + k)])
    r = vx.enclose_system(s, synth.cube(k), depth, vx.make_opts(vx.FP64, timing=True))
    st = r.stats()
    assert st["nodes"].sum(axis=1).max() <= 8192

    def arrays(N):
        return sum(int(n) * (4 + 4 * (d > 0) + 4 * (d + 1 < k)) for d, n in enumerate(N))

    after = list(st["nodes"][1:]) + [r.csf().nodes()[2]]
    want = sum(int(n[-1]) + arrays(n) + arrays(a) for n, a in zip(st["nodes"], after) if n[-1] > 0)
    assert r.timing()["prune_scan"]["work"] == want
