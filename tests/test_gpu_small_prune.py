"""The one-launch prune of small trees on both sides of its size limit (8192 nodes): subdivision
and compaction equal to their definition for one to six variables, with every box, one box and
no box kept; and enclosures through such trees."""
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


def same_tree(vx, c, t, k):
    N, labs, ptrs = oracle.csf(t, k)
    assert c.nodes()[2].tolist() == N.tolist()
    for d in range(1, k + 1):
        lab, ptr = c.export(d)
        assert np.array_equal(lab.cpu().numpy(), labs[d - 1])
        if d < k:
            assert np.array_equal(ptr.cpu().numpy(), ptrs[d - 1].astype(np.int32))
    assert np.array_equal(c.tuples().cpu().numpy(), t)


def nodes(t):
    return sum(np.unique(t[:, :d + 1], axis=0).shape[0] for d in range(t.shape[1]))


@pytest.mark.parametrize("k,level", [(1, 14), (2, 9), (3, 5), (4, 4), (5, 3), (6, 3)])
@pytest.mark.parametrize("most", [8192, 8193, 60])
def test_small_prune_equals_the_definition(vx, k, level, most):
    import torch

    t = synth.random_tuples(k, level, 20000, 3000 + k)
    lo, hi = 1, t.shape[0]
    while lo < hi:  # the longest prefix with at most `most` nodes
        mid = (lo + hi + 1) // 2
        lo, hi = (mid, hi) if nodes(t[:mid]) <= most else (lo, mid - 1)
    t = t[:lo]
    n = t.shape[0]
    c = vx.csf_build(k, level, torch.from_numpy(t).cuda())
    one = np.zeros(n, np.uint8)
    one[n // 2] = 1
    some = (np.random.default_rng(most + k).random(n) < 0.4).astype(np.uint8)
    for keep in (some, one, np.ones(n, np.uint8), np.zeros(n, np.uint8)):
        kept = t[keep != 0]
        d = torch.from_numpy(keep).cuda()
        out, idx = vx.csf_compact(c, d, with_index=True)
        assert np.array_equal(idx.cpu().numpy(), np.flatnonzero(keep))
        if kept.shape[0]:
            same_tree(vx, out, kept, k)
        bits = np.stack(np.meshgrid(*[[0, 1]] * k, indexing="ij"), -1).reshape(1, -1, k)
        kids = (2 * kept[:, None, :] + bits).reshape(-1, k).astype(np.int32)
        kids = kids[np.lexsort(kids.T[::-1])]
        fine = vx.csf_subdivide(c, d)
        assert int(fine.nodes()[2][-1]) == kids.shape[0]
        if kids.shape[0]:
            same_tree(vx, fine, kids, k)


def test_enclosures_through_small_trees(vx):
    """Boxes and codes of enclosures whose levels are all small; a start tree that a small prune
    made (its arrays have room after them) is copied whole."""
    import torch

    polys = [synth.kostlan_poly(3, 6, 3100), synth.kostlan_poly(3, 5, 3101)]
    dom = synth.cube(3)
    ref = oracle.enclose(polys, dom, 5)
    for opts in (vx.make_opts(vx.FP32, host_codes=True), vx.make_opts(vx.FP64)):
        r = vx.enclose(polys, dom, 5, opts)
        assert np.array_equal(vx.Result.decode_codes(r.box_codes(), 3, 5), ref["tuples"])
        assert np.array_equal(r.boxes(), ref["tuples"])
    never = [(np.zeros((1, 3), np.int32), np.array([1.0]))]
    r = vx.enclose(never, dom, 5, vx.make_opts(vx.FP32, host_codes=True))
    assert r.box_codes().shape == (0,) and r.boxes().shape == (0, 3)
    s = vx.System(polys)
    c = vx.csf_full_grid(3, 2)
    start = vx.csf_subdivide(c, vx.csf_eval_level(s, c, dom))
    r = vx.enclose_from(s, start, dom, 5, vx.make_opts(vx.FP64))
    assert np.array_equal(r.boxes(), ref["tuples"])
    torch.cuda.synchronize()
