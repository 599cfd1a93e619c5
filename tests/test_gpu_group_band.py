"""The boxes that the leaf groups leave undecided are those of a bound per pair of leaves: the
bound that a group shares decides what it can, and the rest is evaluated in pairs."""
import numpy as np
import pytest

from paper_2406_09857_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("degrees,rel", [((40,), None), ((40, 37), None), ((40,), [1]),
                                         ((30, 20, 25), [2, 0, 1]), ((40, 40), [3, 4])])
def test_groups_leave_the_pairs_band(vx, degrees, rel):
    polys = [synth.kostlan_poly(3, d, 8700 + 10 * d + i) for i, d in enumerate(degrees)]
    dom = synth.cube(3)
    s = vx.System(polys, rel=rel) if rel else vx.System(polys)
    grid = vx.csf_full_grid(3, 8)
    ref = vx.enclose_from(s, grid, dom, 8, vx.make_opts(vx.FP64))
    band = {}
    try:
        for v in (0, 2, 3, 4):  # pairs; pairs with staged blocks; groups of four and of eight
            vx.autotune(2 + v)
            r = vx.enclose_from(s, grid, dom, 8, vx.make_opts(vx.FP32))
            assert np.array_equal(r.boxes(), ref.boxes()), v
            band[v] = int(r.stats()["recheck"].sum())
    finally:
        vx.autotune(1)
    assert band[0] > 0 and len(set(band.values())) == 1, band
