"""The Taylor form where values overflow: the combination of the derivatives' values equals the
hulls of the four directed endpoint products, summed outward in order, done on the host on the
same values (from the level evaluations of the derivatives as systems of their own)."""
import numpy as np
import pytest

from paper_2406_09857_gb300 import synth

pytestmark = pytest.mark.gpu
MAX = np.finfo(np.float64).max


def add_down(a, b):
    """RD(a + b) elementwise (IEEE for infinite and NaN operands)."""
    with np.errstate(all="ignore"):
        f = np.where(np.maximum(np.abs(a), np.abs(b)) > 2.0 ** 1000, 2.0 ** -4, 1.0)
        x, y = a * f, b * f
        s = x + y
        bb = s - x
        err = (x - (s - bb)) + (y - bb)
        r = np.where(err < 0, np.nextafter(s, -np.inf), s) / f
        finite = np.isfinite(a) & np.isfinite(b)
        r = np.where(finite & (r == np.inf), MAX, r)
        return np.where(finite, r, a + b)


def add_up(a, b):
    return -add_down(-a, -b)


def least(a, b):
    return np.where(b < a, b, a)


def hull(lo, hi, q):
    """[lo, hi] * [-q, q], q a power of two (every product exact)."""
    with np.errstate(all="ignore"):
        p = [lo * -q, lo * q, hi * -q, hi * q]
        mn = least(least(p[0], p[1]), least(p[2], p[3]))
        mx = -least(least(-p[0], -p[1]), least(-p[2], -p[3]))
    return mn, mx


def derivative(e, c, i):
    d = e[:, i] > 0
    e2 = e[d].copy()
    c2 = c[d] * e2[:, i]
    e2[:, i] -= 1
    return e2, c2


@pytest.mark.parametrize("n", [2500, 20001])  # a lane per derivative, a lane per leaf
@pytest.mark.parametrize("k,level", [(2, 9), (3, 6)])
def test_overflowing_taylor_values(vx, k, level, n):
    import torch

    t = synth.random_tuples(k, level, 40000, 8400 + k)
    t = t[::t.shape[0] // n][:n]  # over the whole domain
    assert t.shape[0] == n
    e, _ = synth.uniform_real_poly(k, 6, -10.0, 10.0, 8410 + k)
    c = np.random.default_rng(8420 + k).integers(-9, 10, e.shape[0]) * 2.0 ** 1018
    dom = synth.cube(k, -2.0, 2.0)
    tree = vx.csf_build(k, level, torch.from_numpy(np.ascontiguousarray(t)).cuda())
    w = 4.0 / (1 << level)
    centres = torch.arange(1 << level, dtype=torch.float64, device="cuda") * w + (w / 2 - 2.0)

    def values(poly, at_centre):
        s = vx.System([poly])
        out = (vx.csf_eval_grid(s, tree, [(centres, centres)] * k, vx.FP64, values=True) if at_centre
               else vx.csf_eval_level(s, tree, dom, vx.FP64, values=True))
        return out[1][0].cpu().numpy(), out[2][0].cpu().numpy()

    # multi-indices of order 1 in lexicographic order: 0, e_k, .., e_1
    lo, hi = values((e, c), True)
    for i in reversed(range(k)):
        a, b = hull(*values(derivative(e, c, i), False), w / 2)
        lo, hi = add_down(lo, a), add_up(hi, b)
    keep, glo, ghi = vx.csf_eval_level_taylor(vx.System([(e, c)]), tree, dom, 1, values=True)
    glo, ghi = glo[0].cpu().numpy(), ghi[0].cpu().numpy()
    assert (~np.isfinite(lo)).any() and np.isfinite(lo).any()
    assert np.array_equal(glo, lo, equal_nan=True)
    assert np.array_equal(ghi, hi, equal_nan=True)
    assert np.array_equal(keep.cpu().numpy() == 0, (lo > 0) | (hi < 0))
