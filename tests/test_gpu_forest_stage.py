"""Forests whose depth-1 nodes have at least 64 children per parent stage the parents' blocks in
shared memory (certified binary32): blocks of one fibre group and of several, polynomials of
different lengths in one forest, one and two per system; the boxes are binary64's of each system
alone."""
import numpy as np
import pytest

from paper_2406_09857_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vx():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2406_09857_gb300 import build
    from paper_2406_09857_gb300 import vx as _vx

    build.build()
    _vx.lib()
    return _vx


@pytest.mark.parametrize("degrees", [[(2,), (3,)], [(44,), (45,), (7, 12)], [(60,), (9,), (1,)]])
def test_staged_forest_stage_equals_binary64(vx, degrees):
    depth = 8
    systems = [([synth.kostlan_poly(3, d, 500 + 10 * i + j) for j, d in enumerate(ds)],
                synth.cube(3), depth) for i, ds in enumerate(degrees)]
    got = vx.enclose_batch(systems, vx.make_opts(vx.FP32))
    nodes = sum(np.asarray(r.stats()["nodes"]) for r in got)
    assert any(n[1] >= 16384 and n[1] >= 64 * n[0] for n in nodes)  # the staged form ran
    for (polys, dom, _), r in zip(systems, got):
        one = vx.enclose(polys, dom, depth, vx.make_opts(vx.FP64))
        assert np.array_equal(r.boxes(), one.boxes())
        one.free()
        r.free()
