"""Timed cases of the library: what its users have it do, through its public entry points.

Every case is one call (or the short sequence of calls) of a user's program, on inputs drawn
from a seed.  The families, and what each stands for in real use:

  host      polynomials on the host -> the final boxes' grid codes in the caller's host array
            (vx.enclose): the one-call use of the library, packing and upload included
  enclose   a resident system (vx.System) enclosed again and again, its boxes taken on the
            device: a solver's inner call (vx.enclose_system), in binary64 or certified binary32
  robotics  the manipulator system with interval coefficients, its coefficients perturbed
            (a family of manipulators): few boxes in 4 variables
  control   the control-design system in 6 variables (8 equations, 3 inequalities), perturbed:
            many small polynomials, thin levels, an empty or nearly empty result
  batch     many independent systems of uneven degree and depth in one call
            (vx.enclose_batch), host polynomials to device boxes
  dense     an exactly decided full-grid level of a tensor-product polynomial
            (vx.DensePlan.level_keep)
  taylor    an enclosure with the exclusion test on the Taylor form of order 2, with the
            inclusion test for one equation (hypersurfaces) on request
  values    the interval values and keep flags of one polynomial system on a ragged set of
            boxes (vx.csf_eval_level with values): a caller with its own subdivision loop
  tree      the tree operations of such a loop: build, subdivide, compact (no polynomial)

Coefficient laws and domains are those of paper_2406_09857_gb300/synth.py: Kostlan on [-1,1]^k,
uniform on [-2,2]^k, Gaussian tensors on full grids.  How many boxes survive depends on the
coefficients, so a caller takes them into a buffer with room to spare that it keeps (-1 beyond
the last box).
"""
import functools

import numpy as np
import torch

from paper_2406_09857_gb300 import synth, vx

MODES = {"fp64": vx.FP64, "fp32": vx.FP32}


def listed():
    return [
        # the smallest call: one bivariate curve of degree 20, host to host (the plain workload)
        {"name": "host-k2-d20", "family": "host", "k": 2, "d": 20, "npoly": 1, "depth": 8,
         "law": "integer", "mode": "fp32", "last": False, "first": 0},
        # the robotics system at the depth of its application run, in the default binary64
        {"name": "robotics-fp64", "family": "robotics", "depth": 6, "mode": "fp64", "spread": 0.02},
        # the control-design system: 11 polynomials in 6 variables
        {"name": "control-fp32", "family": "control", "depth": 6, "mode": "fp32",
         "spread": 0.02},
        # an ordinary surface, every level decided as binary64 decides it
        {"name": "surface-fp32", "family": "enclose", "k": 3, "d": 50, "npoly": 1, "depth": 9,
         "law": "kostlan", "mode": "fp32", "last": False, "first": 0},
        # the headline: two surfaces of degree 100 to a 1024^3 grid
        {"name": "curve-fp32", "family": "enclose", "k": 3, "d": 100, "npoly": 2, "depth": 10,
         "law": "kostlan", "mode": "fp32", "last": True, "first": 6},
        # the same from host polynomials to host codes, once per new system, one level coarser
        {"name": "host-curve", "family": "host", "k": 3, "d": 100, "npoly": 2, "depth": 9,
         "law": "kostlan", "mode": "fp32", "last": True, "first": 6},
        # the reference arithmetic on the same system, two levels coarser
        {"name": "curve-fp64", "family": "enclose", "k": 3, "d": 100, "npoly": 2, "depth": 8,
         "law": "kostlan", "mode": "fp64", "last": False, "first": 0},
        # throughput of many small systems (half bivariate, half pairs of surfaces)
        {"name": "batch-256", "family": "batch", "systems": 256, "dmin": 10, "dmax2": 60,
         "dmax3": 40, "lmin": 8, "lmax": 10, "mode": "fp32", "last": True, "sizes": 1},
        # a full grid of 1024^3 boxes, degree 128 in each variable
        {"name": "dense-d128", "family": "dense", "d": 128, "level": 10, "mode": "fp32"},
        # a random-coefficient curve with the tighter exclusion test
        {"name": "taylor-k3-d20", "family": "taylor", "k": 3, "d": 20, "npoly": 2, "depth": 10,
         "c1": False, "mode": "fp32"},
        # one evaluation of scattered boxes with its values, the reference arithmetic
        {"name": "values-fp64", "family": "values", "k": 3, "d": 37, "npoly": 2, "level": 7,
         "boxes": 150000, "mode": "fp64"},
        # one step of a caller's own loop over 4 million boxes
        {"name": "tree-k3", "family": "tree", "k": 3, "level": 9, "boxes": 4000000,
         "share": 0.3},
    ]


def _log(rng, lo, hi):
    """An integer in [lo, hi], uniform in its logarithm."""
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    f = rng.choice(["host", "enclose", "enclose", "robotics", "control", "batch", "dense",
                    "taylor", "values", "tree"])
    mode = rng.choice(["fp32", "fp32", "fp64"])
    if f in ("host", "enclose"):
        k = rng.choice([2, 3, 3])
        npoly = rng.randint(1, k)
        d = _log(rng, 7, 100)
        depth = rng.randint(6, 12) if k == 2 else rng.randint(6, 8 if mode == "fp64" else 10)
        law = rng.choice(["kostlan", "kostlan", "uniform"])
        if npoly == 1 and k == 3:
            depth = min(depth, 8 if mode == "fp64" else 9)
        if law == "uniform":
            depth = min(depth, 7 if mode == "fp64" else 9)
        return {"family": f, "k": k, "d": d, "npoly": npoly, "depth": depth, "law": law,
                "mode": mode, "last": mode == "fp32" and rng.random() < 0.5,
                "first": rng.choice([0, 4, 5, 6])}
    if f == "robotics":
        return {"family": f, "depth": rng.randint(4, 7), "mode": mode,
                "spread": round(rng.uniform(0.001, 0.05), 4)}
    if f == "control":
        return {"family": f, "depth": rng.randint(4, 8), "mode": mode,
                "spread": round(rng.uniform(0.001, 0.05), 4)}
    if f == "batch":
        lmax = rng.randint(7, 9)
        return {"family": f, "systems": _log(rng, 8, 64 if mode == "fp64" else 256),
                "dmin": rng.randint(5, 12),
                "dmax2": rng.randint(20, 60), "dmax3": rng.randint(13, 40), "lmin": lmax - 2,
                "lmax": lmax, "mode": mode, "last": mode == "fp32" and rng.random() < 0.5,
                "sizes": rng.randint(2, 10 ** 6)}
    if f == "dense":
        return {"family": f, "d": _log(rng, 11, 128), "level": rng.randint(6, 9),
                "mode": "fp32"}
    if f == "taylor":
        k = rng.choice([2, 3])
        npoly = rng.randint(1, k)
        return {"family": f, "k": k, "d": _log(rng, 5, 30), "npoly": npoly,
                "depth": rng.randint(6, 8), "c1": npoly == 1 and rng.random() < 0.5,
                "mode": mode}
    if f == "values":
        k, level = rng.choice([2, 3]), rng.randint(4, 9)
        return {"family": f, "k": k, "d": _log(rng, 5, 60), "npoly": rng.randint(1, 3),
                "level": level, "boxes": min(2 ** (k * level - 1), _log(rng, 100, 300000)),
                "mode": mode}
    k = rng.randint(2, 4)
    level = rng.randint(4, 30 // k - 1)
    return {"family": "tree", "k": k, "level": level,
            "boxes": min(2 ** (k * level - 1), _log(rng, 300, 4000000)),
            "share": round(rng.uniform(0.05, 0.95), 3)}


# ---------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------
@functools.lru_cache(maxsize=None)
def _exps(k, d):
    return synth.dense_total_degree(k, d)


@functools.lru_cache(maxsize=None)
def _scale(k, d):
    return synth.kostlan_scale(_exps(k, d), d)


@functools.lru_cache(maxsize=None)
def _tensor_exps(d):
    return synth.dense_per_variable(3, d)


def _stream(seed, part=0):
    return synth.Stream(1000003 * (int(seed) + 1) + 7919 * part)


def _poly(k, d, law, seed, part):
    e, st = _exps(k, d), _stream(seed, part)
    if law == "kostlan":
        return e, st.normal(e.shape[0]) * _scale(k, d)
    if law == "integer":
        return e, st.uniform_int(-1000, 1000, e.shape[0]).astype(np.float64)
    return e, -10.0 + 20.0 * st.unit(e.shape[0])


def _polys(case, seed, law):
    return [_poly(case["k"], case["d"], law, seed, p) for p in range(case["npoly"])]


def _cube(k, law):
    return synth.cube(k, -2.0, 2.0) if law == "uniform" else synth.cube(k)


def _subset(n, total, rng):
    """n of 0 .. total - 1 (n <= total / 2), ascending."""
    got = np.unique(rng.integers(0, total, 2 * n + 64))
    while got.size < n:
        got = np.unique(np.concatenate([got, rng.integers(0, total, n)]))
    return np.sort(rng.choice(got, n, replace=False))


def _tuples(case, seed):
    """case["boxes"] distinct boxes of the level's grid in lexicographic order."""
    k, level = case["k"], case["level"]
    c = _subset(case["boxes"], 2 ** (k * level), np.random.default_rng(int(seed)))
    t = [(c >> (level * (k - 1 - i))) & (2 ** level - 1) for i in range(k)]
    return np.stack(t, axis=1).astype(np.int32)


def _batch_sizes(case):
    """(k, degree, depth) of each system: the same for every seed."""
    st, out = _stream(case["sizes"], 1), []
    for s in range(case["systems"]):
        depth = int(st.uniform_int(case["lmin"], case["lmax"], 1)[0])
        k = 2 if s < case["systems"] // 2 else 3
        out.append((k, int(st.uniform_int(case["dmin"], case["dmax%d" % k], 1)[0]), depth))
    return out


def _room(rows, k):
    return torch.full((int(rows), k), -1, dtype=torch.int32, device="cuda")


def _most(k, npoly, d, depth, law):
    """More boxes than the zero set keeps at the last level."""
    if law == "uniform":
        return 2 ** (k * depth)
    return min(2 ** (k * depth), 4 * _kept(k, npoly, d, depth) + 65536)


def prepare(case, seed):
    f = case["family"]
    st = {"family": f}
    if f in ("host", "enclose"):
        k, law, depth = case["k"], case["law"], case["depth"]
        st["polys"] = _polys(case, seed, law)
        st["domain"], st["depth"] = _cube(k, law), depth
        st["opts"] = vx.make_opts(MODES[case["mode"]], recheck_last=case["last"],
                                  first_level=case["first"], host_codes=f == "host")
        most = _most(k, case["npoly"], case["d"], depth, law)
        if f == "host":
            st["room"] = torch.full((int(most),), -1,
                                    dtype=torch.int32 if k * depth <= 32 else torch.int64)
        else:
            st["room"] = _room(most, k)
            st["system"] = vx.System(st.pop("polys"))
    elif f in ("robotics", "control"):
        s = synth.robotics() if f == "robotics" else synth.automatic()
        nfix = 1 if f == "robotics" else 3  # the sphere, the disks: not perturbed
        polys, his = [], []
        for i, (e, c) in enumerate(s.polys):
            t = np.ones(e.shape[0])
            if i < s.npoly - nfix:
                t += case["spread"] * (2.0 * _stream(seed, i).unit(e.shape[0]) - 1.0)
            polys.append((e, c * t))
            his.append(None if s.his[i] is None else s.his[i] * t)
        st["system"] = vx.System(polys, his=his, rel=s.rel)
        st["domain"], st["depth"] = s.domain, case["depth"]
        st["opts"] = vx.make_opts(MODES[case["mode"]])
        st["room"] = _room(min(2 ** (s.k * case["depth"]), 1 << 22), s.k)
    elif f == "batch":
        st["systems"], most = [], {2: 0, 3: 0}
        for s, (k, d, depth) in enumerate(_batch_sizes(case)):
            polys = [_poly(k, d, "kostlan", seed, 100 + 4 * s + p) for p in range(k - 1)]
            st["systems"].append((polys, synth.cube(k), depth))
            most[k] += _most(k, k - 1, d, depth, "kostlan")
        st["opts"] = vx.make_opts(MODES[case["mode"]], recheck_last=case["last"])
        st["room"] = {k: _room(n, k) for k, n in most.items()}
    elif f == "dense":
        e = _tensor_exps(case["d"])
        c = _stream(seed).normal(e.shape[0])
        st["plan"] = vx.DensePlan(vx.System([(e, c)]), case["level"], synth.cube(3))
        st["opts"] = vx.make_opts(MODES[case["mode"]])
    elif f == "taylor":
        st["system"] = vx.System(_polys(case, seed, "uniform"))
        st["domain"], st["depth"] = _cube(case["k"], "uniform"), case["depth"]
        kw = {"c1": vx.C1_TAYLOR, "c1_level": case["depth"] - 2} if case["c1"] else {}
        if case["mode"] == "fp32":
            kw["small_level_madds"] = 1 << 24
        st["opts"] = vx.make_opts(MODES[case["mode"]], taylor_order=2, **kw)
        most = min(2 ** (case["k"] * case["depth"]), 1 << 22)
        st["room"] = _room(most, case["k"])
        if case["c1"]:
            st["levels"] = np.full(most, -1, np.int32)
            st["certified"] = np.full((most, case["k"]), -1, np.int32)
    elif f == "values":
        st["system"] = vx.System(_polys(case, seed, "kostlan"))
        st["domain"] = synth.cube(case["k"])
        st["csf"] = vx.csf_build(case["k"], case["level"],
                                 torch.from_numpy(_tuples(case, seed)).cuda())
        st["mode"] = MODES[case["mode"]]
    else:
        t = _tuples(case, seed)
        n = t.shape[0]
        keep = np.zeros(n, np.uint8)
        rng = np.random.default_rng(int(seed) + 1)
        keep[rng.permutation(n)[:int(case["share"] * n)]] = 1
        st.update(k=case["k"], level=case["level"], tuples=torch.from_numpy(t).cuda(),
                  keep=torch.from_numpy(keep).cuda())
    return st


def _take(result, room, at=0):
    """The result's boxes into rows at.. of the caller's buffer; the next free row."""
    tree = result.csf()
    n = int(tree.nodes()[2][-1])
    if at + n > room.shape[0]:
        raise RuntimeError("%d boxes do not fit" % n)
    if n and vx.lib().vx_csf_tuples(tree.handle, room[at:].data_ptr(),
                                    torch.cuda.current_stream().cuda_stream) != vx.OK:
        raise RuntimeError(vx.lib().vx_last_error().decode())
    return at + n


def run(st):
    f = st["family"]
    if f == "host":
        r = vx.enclose(st["polys"], st["domain"], st["depth"], st["opts"])
        codes = r.box_codes(copy=False)  # the result's own pinned buffer, until free()
        room = st["room"]
        codes = codes.view(np.int32 if room.dtype == torch.int32 else np.int64)
        room[:codes.shape[0]].copy_(torch.from_numpy(codes))
        r.free()
        return room
    if f in ("enclose", "robotics", "control"):
        r = vx.enclose_system(st["system"], st["domain"], st["depth"], st["opts"])
        n = _take(r, st["room"])
        out = [st["room"], n]
        if f == "control":
            s = r.stats()
            out += [s["tested"], s["kept"]]
        r.free()
        return out
    if f == "batch":
        at = {2: 0, 3: 0}
        for r in vx.enclose_batch(st["systems"], st["opts"]):
            at[r.k] = _take(r, st["room"][r.k], at[r.k])
            r.free()
        return [st["room"][2], st["room"][3], at[2], at[3]]
    if f == "dense":
        return st["plan"].level_keep(st["opts"])[0]
    if f == "taylor":
        r = vx.enclose_system(st["system"], st["domain"], st["depth"], st["opts"])
        n = _take(r, st["room"])
        out = [st["room"], n, r.stats()["kept"]]
        if "levels" in st:
            levels, boxes = r.included()
            st["levels"][:levels.shape[0]] = levels
            st["certified"][:levels.shape[0]] = boxes
            out += [st["levels"], st["certified"]]
        r.free()
        return out
    if f == "values":
        return vx.csf_eval_level(st["system"], st["csf"], st["domain"], st["mode"], values=True)
    c = vx.csf_build(st["k"], st["level"], st["tuples"])
    finer = vx.csf_subdivide(c, st["keep"])
    kept, index = vx.csf_compact(c, st["keep"], with_index=True)
    out = finer.tuples(), kept.tuples(), index
    for t in (c, finer, kept):
        t.free()
    return out


# ---------------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------------
def _terms(k, d):
    n = 1
    for i in range(k):
        n = n * (d + k - i) // (i + 1)
    return n


def _kept(k, npoly, d, level):
    """Boxes kept at a level: 2.5 d boxes across the zero set in each of its normal directions,
    where the grid has so many (measured on the Kostlan surface and curve, within a factor of
    two)."""
    n = 2 ** level
    return float(n) ** (k - npoly) * float(min(n, 2.5 * d)) ** npoly


def _enclose_work(k, npoly, d, depth, host=False, forms=1):
    """Interval Horner of the last variable on every tested box: a multiplication and an addition
    for both ends per coefficient; the work above the leaves is shared by many boxes."""
    tested = sum(2 ** k * _kept(k, npoly, d, lv) for lv in range(depth))
    coefs = npoly * _terms(k, d)
    out = _kept(k, npoly, d, depth)
    return {"bytes": 8 * coefs + out * (4 if host else 4 * k),
            "flops": 4.0 * tested * npoly * d * forms}


def work(case):
    f = case["family"]
    if f in ("host", "enclose"):
        return _enclose_work(case["k"], case["npoly"], case["d"], case["depth"], f == "host")
    if f == "taylor":  # the ten (six) derivatives of order <= 2; few boxes survive
        k, n = case["k"], case["npoly"]
        forms = (k + 1) * (k + 2) // 2
        tested = sum(2 ** k * 2 ** (lv * (k - n)) * 50.0 for lv in range(case["depth"]))
        return {"bytes": 8 * n * _terms(k, case["d"]) + 200.0 * k * 2 ** (case["depth"] * (k - n)),
                "flops": 4.0 * tested * n * forms * case["d"]}
    if f == "robotics":  # 2 polynomials of degree 4 in 4 variables: a few terms per box
        n = 5.0 * 16 ** (case["depth"] - 2)
        return {"bytes": n * 16, "flops": n * 2 * 4 * 5}
    if f == "control":
        n = 64.0 * 6 ** (case["depth"] - 1)
        return {"bytes": n, "flops": n * 11 * 4 * 5}
    if f == "batch":
        each = [_enclose_work(k, k - 1, d, depth) for k, d, depth in _batch_sizes(case)]
        return {q: sum(w[q] for w in each) for q in ("bytes", "flops")}
    if f == "dense":
        n, m = 8.0 ** case["level"], case["d"] + 1
        return {"bytes": n + 8.0 * m ** 3, "flops": 4.0 * n * m}
    if f == "values":
        n, p = case["boxes"], case["npoly"]
        return {"bytes": n * (4.0 * case["k"] + 1 + 16 * p) + 8.0 * p * _terms(case["k"], case["d"]),
                "flops": 4.0 * n * p * case["d"]}
    n, k = case["boxes"], case["k"]  # tuples and flags in; children, kept tuples, indices out
    kept = n * case["share"]
    return {"bytes": n * (4.0 * k + 1) + kept * (2 ** k * 4 * k + 4 * k + 4), "flops": 0}


# ---------------------------------------------------------------------------------------
# values in 64 bits, to nearest
# ---------------------------------------------------------------------------------------
def exact(case, seed):
    """The interval values of the boxes by nested interval Horner, x_1 outermost, in binary64
    rounded to nearest; the other families return whole numbers only."""
    if case["family"] != "values":
        return None
    k, d = case["k"], case["d"]
    if k == 3 and d > 45:
        return None
    t = torch.from_numpy(_tuples(case, seed)).cuda().long()
    w = 2.0 / 2 ** case["level"]
    los, his = [], []
    for e, c in _polys(case, seed, "kostlan"):
        T = np.zeros((d + 1,) * k)
        T[tuple(e.T)] = c
        lo = torch.from_numpy(T).cuda()[None]  # [1, d+1, ..., d+1]: one block, no box yet
        hi = lo
        where = torch.zeros(t.shape[0], dtype=torch.long, device="cuda")
        for i in range(k):
            # the nodes of depth i: distinct (parent block, x_i index)
            node, inv = torch.unique(where * 2 ** case["level"] + t[:, i], return_inverse=True)
            par, ind = node // 2 ** case["level"], node % 2 ** case["level"]
            nl, nh = [], []
            for s in range(0, node.numel(), 4096):
                p, x = par[s:s + 4096], ind[s:s + 4096].double()
                shape = (-1,) + (1,) * (k - 1 - i)
                xl, xh = (-1 + x * w).reshape(shape), (-1 + (x + 1) * w).reshape(shape)
                a, b = lo[p, d], hi[p, d]
                for j in range(d - 1, -1, -1):
                    q = torch.stack([a * xl, a * xh, b * xl, b * xh])
                    a, b = q.amin(0) + lo[p, j], q.amax(0) + hi[p, j]
                nl.append(a)
                nh.append(b)
            lo, hi, where = torch.cat(nl), torch.cat(nh), inv
        los.append(lo[where])
        his.append(hi[where])
    return None, torch.stack(los), torch.stack(his)
