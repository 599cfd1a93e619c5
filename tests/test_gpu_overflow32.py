"""Certified binary32 with values near binary32's largest number: a chain whose partial sums
overflow leaves its boxes to the next tier, so every decision is binary64's, in every launch
variant, in batches, and on domains where the powers of x overflow rather than the
coefficients."""
import numpy as np
import pytest

from paper_2406_09857_gb300 import synth

pytestmark = pytest.mark.gpu

# on [0.8984375, 0.90625] binary64 has [-2.8e36, 4.6e36]; in binary32 both ends of the partial
# sums overflow
CHAIN = [-1.66e38, -3.3e38, 3e38, 3e38]
UNIT = np.array([0.0, 1.0])


def leaf_chain(k, coefs):
    """F(x) = sum_a coefs[a] x_k^a."""
    e = np.zeros((len(coefs), k), np.int32)
    e[:, -1] = np.arange(len(coefs))
    return e, np.array(coefs)


def decisions(vx, s, c, dom, mode):
    return vx.csf_eval_level(s, c, dom, mode).cpu().numpy()


def check(vx, polys, dom, level, k):
    s = vx.System(polys)
    c = vx.csf_full_grid(k, level)
    ref = decisions(vx, s, c, dom, vx.FP64)
    try:
        for v in range(5):
            vx.autotune(2 + v)
            got = decisions(vx, s, c, dom, vx.FP32)
            assert np.array_equal(got, ref), (v, int((got != ref).sum()))
    finally:
        vx.autotune(1)
    return ref


@pytest.mark.parametrize("k", [1, 2, 3])
@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_overflowing_chain(vx, k, sign):
    level = 7 if k < 3 else 6
    dom = np.tile(UNIT, k)
    polys = [leaf_chain(k, [sign * v for v in CHAIN])]
    ref = check(vx, polys, dom, level, k)
    if level == 7:
        assert ref.reshape(-1, 128)[0, 115] == 1  # the box above
    check(vx, polys + [leaf_chain(k, [1e38, -2e38])], dom, level, k)  # two polynomials
    # mirrored: the same chain on x <= 0
    odd = [sign * v * (-1) ** a for a, v in enumerate(CHAIN)]
    check(vx, [leaf_chain(k, odd)], np.tile([-1.0, 0.0], k), level, k)


def test_large_coefficients(vx):
    """Coefficients over the last decades of binary32's range, some of them outside it."""
    kept = tested = 0
    for seed in range(6):
        rng = np.random.default_rng(7000 + seed)
        for k, level in ((2, 7), (3, 5)):
            polys = []
            for f in range(1 + seed % 2):
                e, c = synth.kostlan_poly(k, 3 + seed, 7100 + 10 * seed + f)
                top = 38.4 if seed < 4 else 39.5
                c = np.sign(c) * 10.0 ** rng.uniform(36.0, top, c.shape[0])
                polys.append((e, c))
            ref = check(vx, polys, synth.cube(k), level, k)
            kept += int(ref.sum())
            tested += ref.shape[0]
    assert 0 < kept < tested


@pytest.mark.parametrize("degree,half", [(8, 2.0 ** 16), (20, 64.0), (40, 16.0)])
def test_overflowing_powers(vx, degree, half):
    """Coefficients near 1 (and some that keep the sums small) where x^degree overflows."""
    rng = np.random.default_rng(7300 + degree)
    for k, level in ((2, 7), (3, 5)):
        e = np.zeros((degree + 1, k), np.int32)
        e[:, -1] = np.arange(degree + 1)
        e[:, 0] = degree - e[:, -1]
        c = rng.uniform(-1.0, 1.0, degree + 1)
        check(vx, [(e, c)], synth.cube(k, -half, half), level, k)
        check(vx, [leaf_chain(k, list(c))], synth.cube(k, -half, half), level, k)


def test_overflow_in_batches_and_enclosures(vx):
    systems = [([leaf_chain(2, [s * v for v in CHAIN])], np.tile(UNIT, 2), 7) for s in (1.0, -1.0)]
    systems += [([synth.kostlan_poly(2, 9, 7400)], synth.cube(2), 6)]
    e, c = synth.kostlan_poly(2, 6, 7401)
    systems += [([(e, c * 1e37)], synth.cube(2), 6)]
    ref = [r.boxes() for r in vx.enclose_batch(systems, vx.make_opts(vx.FP64))]
    for last in (False, True):
        opts = vx.make_opts(vx.FP32, recheck_last=last)
        for (p, d, depth), r, a in zip(systems, vx.enclose_batch(systems, opts), ref):
            assert np.array_equal(r.boxes(), a)
            assert np.array_equal(vx.enclose(p, d, depth, opts).boxes(), a)


@pytest.mark.parametrize("rel", [1, 2, 3, 4])
@pytest.mark.parametrize("k", [1, 2])
def test_relations_with_infinite_bounds(vx, rel, k):
    """F < 0 (and the others) where an end and its bound are both infinite: nothing is sure."""
    dom = np.tile(UNIT, k)
    for sign in (1.0, -1.0):
        polys = [leaf_chain(k, [sign * v for v in CHAIN])]
        s = vx.System(polys, rel=[rel])
        c = vx.csf_full_grid(k, 7)
        ref = decisions(vx, s, c, dom, vx.FP64)
        try:
            for v in range(5):
                vx.autotune(2 + v)
                assert np.array_equal(decisions(vx, s, c, dom, vx.FP32), ref), v
        finally:
            vx.autotune(1)
