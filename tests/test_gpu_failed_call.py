"""A call that fails for lack of memory leaves nothing behind: the next one runs."""
import numpy as np
import pytest

from paper_2406_09857_gb300 import synth

pytestmark = pytest.mark.gpu


def test_call_after_a_failed_allocation(vx):
    import torch

    # 2^24 rows of a polynomial with 8 192 entries per row: 2.2 TB of blocks, refused at once
    n = 1 << 24
    t = torch.zeros((n, 2), dtype=torch.int32, device="cuda")
    t[:, 0] = torch.arange(n, device="cuda")
    rows = vx.csf_build(2, 24, t)
    long = vx.System([(np.array([[0, 8191], [1, 0]], np.int32), np.array([1.0, 1.0]))])
    polys = [synth.kostlan_poly(2, 5, 8900)]
    s = vx.System(polys)
    grid = vx.csf_full_grid(2, 6)
    dom = synth.cube(2)
    want = vx.csf_eval_level(s, grid, dom, vx.FP64).cpu().numpy()
    for mode in (vx.FP64, vx.FP32):
        with pytest.raises(RuntimeError, match="bytes"):
            vx.csf_eval_level(long, rows, dom, mode)
        got = vx.csf_eval_level(s, grid, dom, mode).cpu().numpy()
        assert np.array_equal(got, want)
