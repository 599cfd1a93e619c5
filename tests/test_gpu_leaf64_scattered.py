"""The binary64 pair kernel on scattered boxes (warps with few pairs of neighbours go leaf by
leaf) and where its chunks grow: decisions equal to the oracle's."""
import numpy as np
import pytest

import oracle
from paper_2406_09857_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("size", ["smallest", "chunk", "chunk+", "ragged"])
@pytest.mark.parametrize("level,rel", [(14, None), (10, None), (12, [0, 3])])
def test_scattered_boxes(vx, level, rel, size):
    """Level 14: hardly a neighbour; level 10: a few to many in a warp."""
    import torch

    grow = 32 * 128 * torch.cuda.get_device_properties(0).multi_processor_count
    n = {"smallest": 131072, "chunk": grow + grow // 128 - 1, "chunk+": grow + grow // 128,
         "ragged": grow + 77777}[size]
    t = synth.random_tuples(2, level, int(1.6 * n) if level == 10 else int(1.05 * n), 8600 + level)
    if level == 10:  # denser from column to column
        t = t[np.random.default_rng(8).random(t.shape[0]) < 0.4 + 0.6 * (t[:, 0] / 1024.0)]
    t = np.ascontiguousarray(t[:n])
    assert t.shape[0] >= 131072
    polys = [synth.kostlan_poly(2, d, 8610 + d) for d in ((5,) if rel is None else (5, 4))]
    dom = synth.cube(2)
    ref = oracle.eval_csf_gen(polys, dom, level, t, rel=rel)[2]
    s = vx.System(polys, rel=rel) if rel else vx.System(polys)
    c = vx.csf_build(2, level, torch.from_numpy(t).cuda())
    assert np.array_equal(vx.csf_eval_level(s, c, dom, vx.FP64).cpu().numpy(), ref)
