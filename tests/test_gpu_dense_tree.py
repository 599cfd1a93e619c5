"""The dense level's tree from the bit mask and its keep bytes back in grid order: equal to the
full-grid binary64 level for rows of one word, a few and many words, into
buffers of any alignment, with no survivor, and with every box a survivor."""
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


@pytest.mark.parametrize("level", [5, 6, 7, 8])
@pytest.mark.parametrize("what", ["some", "none", "all"])
def test_dense_level_equals_the_full_grid(vx, level, what):
    import torch

    e, c = synth.gaussian_tensor_poly(3, 5, 2900 + level)
    if what == "none":
        c = c * 1e-3
        c[(e == 0).all(axis=1)] = 50.0  # F > 0 on the whole domain
    elif what == "all":
        c = np.where((e.sum(axis=1) == 1), 0.0, c) * 0.0  # F = 0
    sysv = vx.System([(e, c)])
    dom = synth.cube(3)
    grid = vx.csf_full_grid(3, level)
    ref = vx.csf_eval_level(sysv, grid, dom, vx.FP64)
    plan = vx.DensePlan(sysv, level, dom)
    nbox = 1 << (3 * level)
    buf = torch.full((nbox + 9,), 7, dtype=torch.uint8, device="cuda")
    for off in (0, 1, 4):
        for mode in (vx.FP64, vx.FP32):
            keep, n = plan.level_keep(vx.make_opts(mode), keep=buf[off:off + nbox])
            assert torch.equal(keep, ref)
            assert n >= int(ref.sum()) and (what != "none" or n == 0) and (what != "all" or n == nbox)
            assert bool((buf[off + nbox:] == 7).all())  # nothing is written past the end
        buf.fill_(7)
