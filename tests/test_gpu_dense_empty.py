"""A dense level without survivors makes no tree: nothing is launched after the count but the
clearing of the keep flags."""
import numpy as np
import pytest

from paper_2406_09857_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("level", [5, 6, 7, 8, 9])
def test_dense_level_without_survivors(vx, level):
    import torch

    e, c = synth.gaussian_tensor_poly(3, 3, 2950 + level)
    first = (e == 0).all(axis=1)
    s = vx.System([(e, np.where(first, 10.0 + np.abs(c).sum(), c))])
    dom = synth.cube(3)
    plan = vx.DensePlan(s, level, dom)
    keep = torch.full((1 << (3 * level),), 7, dtype=torch.uint8, device="cuda")
    opts = vx.make_opts(vx.FP32)
    plan.level_keep(opts, keep=keep)
    before = vx.kernel_launches()
    _, n = plan.level_keep(opts, keep=keep)
    launches = vx.kernel_launches() - before
    assert n == 0 and not bool(keep.any())
    mask = plan.prefilter()
    before = vx.kernel_launches()
    plan.prefilter(mask)
    assert launches == vx.kernel_launches() - before + 2  # the rows' and the slabs' counts
    # one box kept: F changes sign there only (a linear factor at a corner of the domain)
    e1 = np.array([[0, 0, 0], [1, 0, 0], [0, 1, 0], [0, 0, 1]], np.int32)
    w = 2.0 / (1 << level)
    s1 = vx.System([(e1, np.array([3.0 - 0.5 * w, 1.0, 1.0, 1.0]))])
    p1 = vx.DensePlan(s1, level, dom)
    ref = vx.csf_eval_level(s1, vx.csf_full_grid(3, level), dom, vx.FP64)
    k1, _ = p1.level_keep(opts)
    assert int(ref.sum()) > 0 and torch.equal(k1, ref)
