"""Batches from several host threads at once: each thread's forests need their own amount of
shared memory, and none of them lowers what another one's launch may use."""
import threading

import numpy as np
import pytest

from paper_2406_09857_gb300 import synth

pytestmark = pytest.mark.gpu


def long_chain(n, c):
    """x_2^n + x_1 - c: a leaf block of n + 1 entries."""
    return np.array([[0, n], [1, 0], [0, 0]], np.int32), np.array([1.0, 1.0, -c])


def test_batches_of_different_degrees_at_once(vx):
    import torch

    dom = synth.cube(2)
    small = [([synth.kostlan_poly(2, 4, 8000 + i)], dom, 5) for i in range(3)]
    large = [([long_chain(4500, 0.25 + 0.1 * i)], dom, 5) for i in range(3)]
    opts = vx.make_opts(vx.FP32)
    ref = {id(b): [r.boxes() for r in vx.enclose_batch(b, vx.make_opts(vx.FP64))]
           for b in (small, large)}
    errors = []

    def work(batch):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(150):
                    got = vx.enclose_batch(batch, opts, nworkers=1)
                    for r, b in zip(got, ref[id(batch)]):
                        assert np.array_equal(r.boxes(), b)
                        r.free()
        except Exception as e:  # noqa: BLE001
            errors.append(repr(e))

    threads = [threading.Thread(target=work, args=(b,)) for b in (small, large, small, large)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[:2]
