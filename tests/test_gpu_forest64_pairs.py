"""The binary64 pair kernel of a forest: a batch that is certain to be large enough for it, against
the CPU oracle."""
import numpy as np
import pytest

import oracle
from paper_2406_09857_gb300 import synth

pytestmark = pytest.mark.gpu


def test_forest_of_binary64_pairs_equals_the_oracle(vx):
    systems = [([synth.kostlan_poly(3, 4, 8300)], synth.cube(3), 7),
               ([synth.kostlan_poly(3, 6, 8301)], synth.cube(3), 6),
               ([synth.kostlan_poly(3, 5, 8302), synth.kostlan_poly(3, 3, 8303)], synth.cube(3), 7)]
    rs = vx.enclose_batch(systems, vx.make_opts(vx.FP64))
    tested = sum(np.pad(r.stats()["tested"], (0, 8 - len(r.stats()["tested"]))) for r in rs)
    assert tested.max() >= 131072  # a level's leaves over the forest
    for (polys, dom, depth), r in zip(systems, rs):
        ref = oracle.enclose(polys, dom, depth)
        assert np.array_equal(r.boxes(), ref["tuples"])
        assert np.array_equal(r.stats()["tested"], ref["tested"])
