"""The certified binary32 leaves on groups of neighbouring leaves (points of the boxes, then the
one end that is left): decisions equal to the oracle's, bit for bit, where the groups can go wrong:
chains of every length modulo the unrolling, groups that straddle parents and the sign of x_k,
leaves that are no neighbours, partial groups, inequalities, and several polynomials."""
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


def boxes(k, level, shape, seed):
    """Lex-sorted box indices: "full" grid, "random" subset, or "runs" of neighbours of uneven
    length and position in every column (x_k)."""
    side = 1 << level
    if shape == "random":
        return synth.random_tuples(k, level, side ** k // 3, seed)
    g = np.stack(np.meshgrid(*[np.arange(side)] * k, indexing="ij"), -1).reshape(-1, k)
    if shape == "full":
        return g.astype(np.int32)
    rng = np.random.default_rng(seed)
    first = rng.integers(0, side, side ** (k - 1)).repeat(side)
    count = rng.integers(0, side, side ** (k - 1)).repeat(side)
    return g[(g[:, -1] >= first) & (g[:, -1] < first + count)].astype(np.int32)


@pytest.mark.parametrize("shape", ["full", "runs", "random"])
@pytest.mark.parametrize("degrees,rel,domain", [
    ((0,), None, (-1, 1)), ((1,), None, (-1, 1)), ((2, 3), None, (-1, 1)),
    ((4, 5, 6), None, (-1, 1)), ((7,), None, (-0.75, 1.25)), ((9, 8), [0, 1], (-1, 1)),
    ((6, 7, 3), [2, 0, 0], (-2, 2)), ((12, 17), None, (0, 1))])
def test_leaf_groups_decide_as_the_oracle(vx, degrees, rel, domain, shape):
    import torch

    for k, level in ((2, 5), (3, 4)):
        polys = [synth.kostlan_poly(k, d, 2100 + 10 * i + d) for i, d in enumerate(degrees)]
        dom = synth.cube(k, *[float(v) for v in domain])
        t = boxes(k, level, shape, 2200 + level)
        ref = oracle.eval_csf_gen(polys, dom, level, t, rel=rel)[2]
        s = vx.System(polys, rel=rel) if rel else vx.System(polys)
        c = vx.csf_build(k, level, torch.from_numpy(t).cuda())
        try:
            for v in (3, 4):
                vx.autotune(2 + v)
                keep = vx.csf_eval_level(s, c, dom, vx.FP32).cpu().numpy()
                assert np.array_equal(keep, ref), (k, v)
        finally:
            vx.autotune(1)


@pytest.mark.parametrize("shape", ["full", "runs", "random"])
@pytest.mark.parametrize("degrees,rel,domain", [
    ((0,), None, (-1, 1)), ((2, 3), None, (-1, 1)), ((7, 4), [3, 0], (-0.75, 1.25)),
    ((5, 6, 3), [2, 4, 1], (-2, 2))])
def test_binary64_pairs_decide_as_the_oracle(vx, degrees, rel, domain, shape):
    """The binary64 leaves in pairs (levels of 2^17 leaves and more), the same way; the last
    set is just below that size (one leaf per thread)."""
    import torch

    for k, level, cut in ((2, 10, None), (3, 7, None), (2, 10, 131071)):
        polys = [synth.kostlan_poly(k, d, 2300 + 10 * i + d) for i, d in enumerate(degrees)]
        dom = synth.cube(k, *[float(v) for v in domain])
        t = boxes(k, level, shape, 2400 + level)[:cut]
        assert cut or t.shape[0] >= 131072
        ref = oracle.eval_csf_gen(polys, dom, level, t, rel=rel)[2]
        s = vx.System(polys, rel=rel) if rel else vx.System(polys)
        c = vx.csf_build(k, level, torch.from_numpy(t).cuda())
        assert np.array_equal(vx.csf_eval_level(s, c, dom, vx.FP64).cpu().numpy(), ref), (k, cut)


def test_binary64_forest_pairs_equal_single_runs(vx):
    """A forest large enough for the pairs, one system of no box among them."""
    dom = synth.cube(3)
    systems = [([synth.kostlan_poly(3, d, 2500 + 3 * d), synth.kostlan_poly(3, d, 2501 + 3 * d)],
                dom, 7) for d in (4, 9, 12)]
    never = (np.zeros((1, 3), np.int32), np.array([1.0]))  # F = 1: no box is kept
    systems.insert(1, ([never, never], dom, 7))
    rs = vx.enclose_batch(systems, vx.make_opts(vx.FP64))
    assert max(r.stats()["tested"].max() for r in rs) > 0
    for (polys, d, depth), r in zip(systems, rs):
        ref = vx.enclose(polys, d, depth, vx.make_opts(vx.FP64))
        assert np.array_equal(r.boxes(), ref.boxes())
        assert np.array_equal(r.stats()["kept"], ref.stats()["kept"])
