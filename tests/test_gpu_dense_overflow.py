"""The tensor-core prefilter where a box's midpoint overflows binary32: such a box is not
excluded, so the dense level's keep flags are binary64's."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_dense_level_with_overflowing_midpoints(vx, axis, sign):
    """-2.5e38 (1 + x) + 3.3e38 (x^8 + x^9) has a zero near x = 0.96, where the first two terms
    alone pass binary32's largest number (the last two come in another step of the product)."""
    e = np.zeros((4, 3), np.int32)
    e[:, axis] = [0, 1, 8, 9]
    c = sign * np.array([-2.5e38, -2.5e38, 3.3e38, 3.3e38])
    s = vx.System([(e, c)])
    dom = np.array([0.0, 1.0] * 3)
    ref = vx.csf_eval_level(s, vx.csf_full_grid(3, 6), dom, vx.FP64).cpu().numpy()
    assert 0 < ref.sum() < ref.shape[0]
    plan = vx.DensePlan(s, 6, dom)
    mask = vx.mask_to_bool(plan.prefilter(), 1 << 18).cpu().numpy()
    assert not np.any(ref.astype(bool) & ~mask)
    for mode in (vx.FP64, vx.FP32):
        keep, _ = plan.level_keep(vx.make_opts(mode))
        assert np.array_equal(keep.cpu().numpy(), ref)
    mid, rad = [x.cpu().numpy().astype(np.float64) for x in plan.values()]
    assert np.all(np.isinf(rad[~np.isfinite(mid)]))
