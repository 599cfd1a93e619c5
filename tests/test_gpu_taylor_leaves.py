"""The Taylor form's leaf kernels on both sides of the line between a lane per derivative and
a lane per leaf: values, C0 and C1 equal to the oracle's bit for bit, binary32's decisions too; with
values that overflow (where the binary64 steps take the endpoint product that finite values
make extremal, and the oracle the hull of all four), the two kernels equal one another."""
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


@pytest.mark.parametrize("k,level,order,n", [(1, 6, 3, 1), (2, 9, 3, 16384), (2, 9, 3, 16385),
                                             (3, 6, 2, 9), (3, 6, 1, 16384), (3, 6, 2, 20001)])
def test_taylor_leaves_equal_the_oracle(vx, k, level, order, n):
    import torch

    t = synth.random_tuples(k, level, 2 * n + 40, 2800 + level)[:n]
    assert t.shape[0] == n
    dom = synth.cube(k, -2.0, 2.0)
    polys = [synth.uniform_real_poly(k, 6, -10.0, 10.0, 2810 + f) for f in range(2)]
    c = vx.csf_build(k, level, torch.from_numpy(np.ascontiguousarray(t)).cuda())
    lo, hi, keep = oracle.taylor_boxes(polys, dom, level, order, t)
    s = vx.System(polys)
    got = [x.cpu().numpy() for x in vx.csf_eval_level_taylor(s, c, dom, order, values=True)]
    assert np.array_equal(got[0], keep)
    assert np.array_equal(got[1], lo) and np.array_equal(got[2], hi)
    assert np.array_equal(vx.csf_taylor_level(s, c, dom, order, vx.FP32)[0].cpu().numpy(), keep)
    if order >= 2:
        one = vx.System(polys[:1])
        ref = oracle.c1_boxes(polys[0], dom, level, oracle.C1_TAYLOR, t, order)
        for mode in (vx.FP64, vx.FP32):
            inc = vx.csf_taylor_level(one, c, dom, order, mode, c1=True)[1].cpu().numpy()
            assert np.array_equal(inc, ref)


@pytest.mark.parametrize("k,level,order", [(2, 9, 3), (3, 6, 2)])
def test_taylor_leaf_kernels_agree_on_overflow(vx, k, level, order):
    import torch

    t = synth.random_tuples(k, level, 40000, 2800 + level)[:20001]
    polys = [(e, c * 1e306) for e, c in
             (synth.uniform_real_poly(k, 6, -10.0, 10.0, 2810 + f) for f in range(2))]
    dom = synth.cube(k, -2.0, 2.0)
    s = vx.System(polys)

    def values(t):
        c = vx.csf_build(k, level, torch.from_numpy(np.ascontiguousarray(t)).cuda())
        return [x.cpu().numpy() for x in vx.csf_eval_level_taylor(s, c, dom, order, values=True)]

    whole, a, b = values(t), values(t[:9000]), values(t[9000:])
    assert np.isnan(whole[1]).any()
    for w, x, y in zip(whole, a, b):
        assert np.array_equal(w, np.concatenate([x, y], axis=-1), equal_nan=w.dtype.kind == "f")
