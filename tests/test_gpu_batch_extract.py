"""A batch's final trees, taken out of a level's forest in one launch: trees of very different
sizes finishing at one level and at several, a tree whose boxes all go before its depth, one
whose boxes all go at it, and depth 0; each equal to the CSF of its own system's enclosure."""
import numpy as np
import pytest

import oracle
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


def sphere(k, r2):
    """x_1^2 + .. + x_k^2 - r2"""
    e = np.vstack([2 * np.eye(k, dtype=np.int32), np.zeros((1, k), np.int32)])
    return e.astype(np.int32), np.array([1.0] * k + [-float(r2)])


@pytest.mark.parametrize("k,top", [(1, 9), (2, 9), (3, 6), (4, 4)])
@pytest.mark.parametrize("mode", ["FP64", "FP32"])
def test_batch_trees_equal_single_enclosures(vx, k, top, mode):
    systems = [([sphere(k, r2)], synth.cube(k), depth)
               for r2, depth in [(0.5, top), (-1.0, top), (0.0, top), (0.7, top - 2), (0.3, 0),
                                 (1e-4, top), (-1.0, 0), (0.9, top)]]
    opts = vx.make_opts(getattr(vx, mode))
    for (polys, dom, depth), r in zip(systems, vx.enclose_batch(systems, opts)):
        one = vx.enclose(polys, dom, depth, opts)
        boxes = one.boxes()
        assert np.array_equal(r.boxes(), boxes)
        c = r.csf()
        N, labs, ptrs = oracle.csf(boxes, k) if boxes.shape[0] else (np.zeros(k, int), None, None)
        assert c.nodes()[2].tolist() == N.tolist()
        for d in range(1, k + 1 if boxes.shape[0] else 1):
            lab, ptr = c.export(d)
            assert np.array_equal(lab.cpu().numpy(), labs[d - 1])
            if d < k:
                assert np.array_equal(ptr.cpu().numpy(), ptrs[d - 1].astype(np.int32))
        one.free()
        r.free()
