"""Tree builds and index tuples with vector loads and stores: equal to the definition for one to
six variables, at sizes around a thread's eight tuples, a warp's 128 leaves and a scan tile, from
and into buffers that do and do not start on 16 bytes; bad tuples are refused wherever they are."""
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


@pytest.mark.parametrize("k,level", [(1, 16), (2, 9), (3, 6), (4, 5), (5, 4), (6, 3)])
def test_build_and_tuples(vx, k, level):
    import torch

    full = synth.random_tuples(k, level, 30000, 3200 + k)
    stream = torch.cuda.current_stream().cuda_stream
    for n in (1, 7, 8, 9, 127, 128, 129, 2047, 2049, 16385):
        t = full[:n]
        assert t.shape[0] == n
        N, labs, ptrs = oracle.csf(t, k)
        for off in (0, 1):
            buf = torch.zeros(n * k + 4, dtype=torch.int32, device="cuda")
            buf[off:off + n * k] = torch.from_numpy(np.ascontiguousarray(t)).cuda().view(-1)
            c = vx.csf_build(k, level, buf[off:off + n * k].view(n, k))
            assert c.nodes()[2].tolist() == N.tolist()
            for d in range(1, k + 1):
                lab, ptr = c.export(d)
                assert np.array_equal(lab.cpu().numpy(), labs[d - 1])
                if d < k:
                    assert np.array_equal(ptr.cpu().numpy(), ptrs[d - 1].astype(np.int32))
            out = torch.full((n * k + 4,), -7, dtype=torch.int32, device="cuda")
            assert vx.lib().vx_csf_tuples(c.handle, out[off:].data_ptr(), stream) == vx.OK
            out = out.cpu().numpy()
            assert np.array_equal(out[off:off + n * k].reshape(n, k), t)
            assert (out[:off] == -7).all() and (out[off + n * k:] == -7).all()


@pytest.mark.parametrize("k,level", [(1, 16), (3, 6), (6, 3)])
def test_bad_tuples_are_refused(vx, k, level):
    import torch

    t = synth.random_tuples(k, level, 9000, 3300 + k)[:4000]
    for at in (0, 1, 7, 8, 255, 2048, 3999):
        for kind in ("range", "negative", "order", "twice"):
            bad = t.copy()
            if kind == "range":
                bad[at, k - 1] = 1 << level
            elif kind == "negative":
                bad[at, 0] = -1
            elif at == 0:
                continue
            elif kind == "order":
                bad[[at - 1, at]] = bad[[at, at - 1]]
            else:
                bad[at] = bad[at - 1]
            with pytest.raises(vx.VxError) as e:
                vx.csf_build(k, level, torch.from_numpy(bad).cuda())
            assert e.value.code == vx.EINVAL
