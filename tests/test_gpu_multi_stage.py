"""One launch for a depth's stage of several polynomials: values and decisions equal to the
oracle's where some of a system's polynomials share the launch and others are too large for it,
for two to four variables, every arithmetic, and a level too large for any to share."""
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


# (k, level, boxes, degrees): 2^21 (node, fibre) items is the line.  In the second case the
# depth-2 stage of degree 40 (61 000 nodes, 41 fibres) is above it and the other two below, in
# the third one polynomial is left alone, in the last all are above it.
@pytest.mark.parametrize("k,level,n,degrees", [
    (2, 6, 900, (3, 8, 5)), (3, 8, 200000, (3, 40, 4)), (3, 8, 200000, (40, 2)),
    (4, 3, 1000, (3, 1, 4, 0)), (3, 9, 300000, (14, 13))])
def test_shared_stage_launches_equal_the_oracle(vx, k, level, n, degrees):
    import torch

    polys = [synth.kostlan_poly(k, d, 2600 + 10 * i + d) for i, d in enumerate(degrees)]
    dom = synth.cube(k)
    t = synth.random_tuples(k, level, n, 2700 + level)
    lo, hi, keep, _ = oracle.eval_csf_gen(polys, dom, level, t)
    s = vx.System(polys)
    c = vx.csf_build(k, level, torch.from_numpy(t).cuda())
    got, glo, ghi = (x.cpu().numpy() for x in vx.csf_eval_level(s, c, dom, vx.FP64, values=True))
    assert np.array_equal(got, keep) and np.array_equal(glo, lo) and np.array_equal(ghi, hi)
    try:
        for v in (0, 1, 2):  # the forced launch variants
            vx.autotune(2 + v)
            assert np.array_equal(vx.csf_eval_level(s, c, dom, vx.FP64).cpu().numpy(), keep)
            assert np.array_equal(vx.csf_eval_level(s, c, dom, vx.FP32).cpu().numpy(), keep)
            m, mlo, mhi = vx.csf_eval_level(s, c, dom, vx.FP32_MIDRAD, values=True)
            assert (mlo.cpu().numpy() <= lo).all() and (mhi.cpu().numpy() >= hi).all()
            assert (m.cpu().numpy() >= keep).all()
    finally:
        vx.autotune(1)
