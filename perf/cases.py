"""What a user of the depth library has it compute, as measurable cases.

Every case is one call (or one burst of calls) through the public binding:
``Context.depth``, ``Context.depth_batched`` or ``Stream.submit`` / ``wait``.
The sizes are those of the seeded workloads (W1 ... W7) and of the ranges they
are drawn from; the data are integers as the library takes them: uniform,
rounded Gaussian, or rounded Student-t with copied rows and rows on one
hyperplane.  Query points are, unless the case says otherwise, data rows and
uniform points of the data's bounding box, half and half.
"""
from math import comb, exp, log

import numpy as np
import torch

from paper_1409_3901_gb300 import tukey

ALGORITHMS = {"rcom": tukey.TD_ALG_RCOM, "adia": tukey.TD_ALG_ADIA}
# (query, subset, point) triples of the largest drawn call: below the listed
# p = 5 call with ties (256 queries, C(200, 3) subsets, 200 points)
MOST = 3e10


def _depth(name, p, n, m, data, **more):
    case = {"name": name, "call": "depth", "p": p, "n": n, "m": m, "data": data, "lim": 127,
            "queries": "half", "host": False, "algorithm": "rcom", "early_exit": False}
    case.update(more)
    return case


def listed():
    return [
        # one point scored against a small sample, host arrays in and out: the
        # smallest call there is, where copies and launches are what counts
        _depth("one_query_host", 3, 300, 1, "uniform", host=True),
        # the small plain-method configuration (W1)
        _depth("small_p3", 3, 300, 16, "uniform"),
        # the bivariate case alone, many queries (W6): one sweep a query
        _depth("bivariate_many", 2, 2000, 16384, "gaussian"),
        # the depth of every row within its own sample (outlier ranking), with
        # coordinates of 15 bits instead of 8
        _depth("own_depths_p3", 3, 1000, 1000, "gaussian", lim=16000, queries="own"),
        # the benchmark's configuration (W2)
        _depth("batch_p4", 4, 1000, 64, "gaussian"),
        # copies and a common hyperplane, many queries (W4)
        _depth("ties_p5", 5, 200, 256, "t3ties"),
        # the largest dimension, at the largest n the request stream gives it
        _depth("largest_p6", 6, 120, 8, "uniform"),
        # a query that only has to reach the answer: stops at depth zero
        _depth("early_exit_p4", 4, 641, 40, "gaussian", early_exit=True),
        # Algorithm 3 on the benchmark's configuration
        _depth("adaptive_p4", 4, 1000, 64, "gaussian", algorithm="adia"),
        # coordinates over the whole int32 range: the 256-bit path
        _depth("full_range_p3", 3, 150, 16, "int32"),
        # independent datasets of uneven n and p in one call (W3)
        {"name": "datasets_batched", "call": "batched", "sets": 16, "m": 16, "most": 4e9},
        # requests submitted as they come and waited for (W5)
        {"name": "request_stream", "call": "stream", "requests": 16, "most": 3e8},
    ]


def _log_int(rng, lo, hi):
    return int(round(exp(rng.uniform(log(lo), log(hi)))))


def _triples(p, n, m):
    return float(comb(n, max(p - 2, 0))) * n * m


def draw(rng):
    kind = rng.choice(["depth"] * 6 + ["adia", "early", "int32", "batched", "stream"])
    if kind == "batched":
        return {"call": "batched", "sets": rng.randint(2, 16), "m": rng.randint(1, 16), "most": 1e9}
    if kind == "stream":
        return {"call": "stream", "requests": rng.randint(1, 16), "most": 2e8}
    if kind == "int32":
        p = rng.choice([2, 3])
        return _depth(None, p, rng.randint(20, 150), rng.randint(1, 16), "int32", host=rng.random() < 0.5)
    p = rng.randint(2, 6) if kind == "depth" else rng.randint(3, 5)
    most = MOST / 4 if kind == "depth" else MOST / 16
    while True:
        n = _log_int(rng, 16, 2000) + rng.randint(0, 47)
        m = _log_int(rng, 1, 4000 if p == 2 else 512)
        if _triples(p, n, m) <= most:
            break
    return _depth(None, p, n, m, rng.choice(["uniform", "gaussian", "t3ties"]),
                  lim=rng.choice([12, 127, 127, 1000]), queries=rng.choice(["half", "half", "own", "centre"]),
                  host=rng.random() < 0.3, early_exit=kind == "early",
                  algorithm="adia" if kind == "adia" else "rcom")


def _rows(kind, n, p, lim, g):
    if kind == "int32":
        return g.integers(-2 ** 31, 2 ** 31, (n, p)).astype(np.int32)
    if kind == "uniform":
        return g.integers(-lim, lim + 1, (n, p)).astype(np.int32)
    if kind == "gaussian":
        return np.clip(np.rint(g.standard_normal((n, p)) * (lim * 40 / 127)), -lim, lim).astype(np.int32)
    # Student-t with 3 degrees of freedom, a tenth of the rows copies of
    # others, a twentieth on one hyperplane
    x = np.clip(np.rint(g.standard_t(3, (n, p)) * (lim * 20 / 127)), -lim, lim).astype(np.int32)
    perm = g.permutation(n)
    k, h = n // 10, n // 20
    x[perm[:k]] = x[perm[k:2 * k]]
    plane = perm[2 * k:2 * k + h]
    x[plane, p - 1] = np.clip(x[plane, :p - 1].sum(axis=1), -lim, lim)
    return x


def _points(how, x, m, g):
    lo, hi = x.min(axis=0).astype(np.int64), x.max(axis=0).astype(np.int64)
    n = len(x)
    if how == "own":
        return x[np.arange(m) % n].copy()
    if how == "centre":
        mid, r = (lo + hi) // 2, (hi - lo) // 4
        return g.integers(mid - r, mid + r + 1, (m, x.shape[1])).astype(np.int32)
    rows = x[g.permutation(n)[np.arange(m // 2) % n]]
    return np.concatenate([rows, g.integers(lo, hi + 1, (m - m // 2, x.shape[1])).astype(np.int32)])


def _dataset(case, seed):
    g = np.random.default_rng([seed, 1409])
    x = _rows(case["data"], case["n"], case["p"], case["lim"], g)
    return x, _points(case["queries"], x, case["m"], g)


def _shape(g, dims, low, high, most):
    p = int(g.choice(dims))
    n = int(round(exp(g.uniform(log(low), log(high)))))
    while comb(n, p - 2) * n > most:
        n -= 1
    return n, p


def _sets(case, seed):
    """Datasets of p in {3, 4, 5} and log-uniform n (W3's); which shapes they
    have is the case's, the values the seed's."""
    shapes, g = np.random.default_rng(1409), np.random.default_rng([seed, 1410])
    out = []
    for _ in range(case["sets"]):
        n, p = _shape(shapes, [3, 4, 5], 100, 2000, case["most"])
        x = _rows("gaussian" if shapes.random() < 0.5 else "uniform", n, p, 127, g)
        out.append((x, _points("half", x, case["m"], g)))
    return out


def _requests(case, seed):
    """Requests of p in {3, ..., 6}, n in [50, 1000], 1 to 64 queries (W5's)."""
    shapes, g = np.random.default_rng(1411), np.random.default_rng([seed, 1412])
    out = []
    for _ in range(case["requests"]):
        n, p = _shape(shapes, [3, 4, 5, 6], 50, 1000, case["most"])
        x = _rows("uniform", n, p, 127, g)
        out.append((x, _points("half", x, int(shapes.integers(1, 65)), g)))
    return out


def _device(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def prepare(case, seed):
    if case["call"] == "stream":
        ctx = tukey.Context(0)
        return {"call": "stream", "requests": _requests(case, seed), "stream": ctx.stream(1 << 30)}
    if case["call"] == "batched":
        return {"call": "batched", "ctx": tukey.Context(0, device_pointers=True),
                "sets": [(_device(x), _device(z)) for x, z in _sets(case, seed)]}
    x, z = _dataset(case, seed)
    opts = {"algorithm": ALGORITHMS[case["algorithm"]], "early_exit": case["early_exit"]}
    if case["host"]:
        return {"call": "depth", "ctx": tukey.Context(0, **opts), "x": x, "z": z}
    return {"call": "depth", "ctx": tukey.Context(0, device_pointers=True, **opts), "x": _device(x), "z": _device(z)}


def run(state):
    if state["call"] == "stream":
        s = state["stream"]
        tickets = [s.submit(x, z) for x, z in state["requests"]]
        return [s.wait(t) for t in tickets]
    if state["call"] == "batched":
        return state["ctx"].depth_batched(state["sets"])
    return state["ctx"].depth(state["x"], state["z"])


def _work(x_shape, m, algorithm="rcom", early_exit=False, wide=False):
    n, p = x_shape
    if wide:  # every hyperplane through p - 1 points: the side of every point
        flops = 2.0 * p * comb(n, p - 1) * n * m
    elif early_exit or algorithm == "adia":  # the counts of the data directions, at least
        flops = 2.0 * p * n * n * m
    else:
        # a point in a sweep: two multiply-adds onto the last two coordinates
        # of the quotient, one operation to place it, one to count it
        flops = 6.0 * _triples(p, n, m)
    return 4.0 * (n * p + m * p + m), flops


def work(case):
    if case["call"] == "depth":
        parts = [_work((case["n"], case["p"]), case["m"], case["algorithm"], case["early_exit"],
                       case["data"] == "int32")]
    else:
        sets = _sets(case, 0) if case["call"] == "batched" else _requests(case, 0)
        parts = [_work(x.shape, len(z)) for x, z in sets]
    return {"bytes": sum(b for b, _ in parts), "flops": sum(f for _, f in parts)}


def _line(v):
    """The fewest points strictly on one side of 0 on a line through it."""
    lead = v[np.arange(len(v)), (v != 0).argmax(axis=1)] if len(v) else np.zeros(0)
    first = v[0] if len(v) else None
    side = np.sign(lead) if first is None else np.sign((v * first).sum(axis=1))
    return int(min((side > 0).sum(), (side < 0).sum()))


def _plane(v):
    """The fewest points strictly on one side of a line through 0, over all
    lines in general position, for nonzero integer points of the plane."""
    best = len(v)
    for a, b in v:
        s = np.sign(a * v[:, 1] - b * v[:, 0])
        on = v[s == 0]
        best = min(best, int(min((s > 0).sum(), (s < 0).sum())) + _line(on))
    return best


def _space(x, z):
    """T(z) for p = 3: over the planes through z and two points, the fewest
    points strictly on one side plus the same count inside the plane."""
    v = x.astype(np.int64) - z.astype(np.int64)
    zero = int((v == 0).all(axis=1).sum())
    v = v[(v != 0).any(axis=1)]
    i, j = np.triu_indices(len(v), 1)
    normal = np.cross(v[i], v[j])
    normal = normal[(normal != 0).any(axis=1)]
    side = normal.astype(np.float64) @ v.T.astype(np.float64)  # below 2^53: exact
    pos, neg = (side > 0).sum(axis=1), (side < 0).sum(axis=1)
    strict = np.minimum(pos, neg)
    best = len(v)
    for k in np.argsort(strict, kind="stable"):
        if strict[k] >= best:
            break
        drop = int((normal[k] != 0).argmax())
        best = min(best, int(strict[k]) + _plane(np.delete(v[side[k] == 0], drop, axis=1)))
    return zero + best


def _flat(x, z):
    """T(z) for p = 2 and every row of z: lines sorted by direction.  The key
    y1 / (|y1| + |y2|) of the direction turned to the upper half plane is one
    rounding of a quotient of small integers, so equal directions have equal
    keys and different ones different keys."""
    out = []
    for part in np.array_split(z, max(1, len(z) // 256)):
        v = x[None].astype(np.int64) - part[:, None].astype(np.int64)
        nonzero = (v != 0).any(axis=2)
        up = (v[..., 1] > 0) | ((v[..., 1] == 0) & (v[..., 0] > 0))
        h = np.where(up[..., None], v, -v).astype(np.float64)
        with np.errstate(invalid="ignore"):
            key = np.where(nonzero, -h[..., 0] / (np.abs(h[..., 0]) + h[..., 1]), 9.0)
        order = np.argsort(key, axis=1, kind="stable")
        key = np.take_along_axis(key, order, 1)
        step = np.take_along_axis(np.where(nonzero, np.where(up, -1, 1), 0), order, 1)
        count = nonzero.sum(axis=1)
        walk = (up & nonzero).sum(axis=1)[:, None] + np.cumsum(step, axis=1)
        last = np.concatenate([key[:, 1:] != key[:, :-1], np.ones((len(part), 1), bool)], axis=1)
        value = np.where(last, np.minimum(walk, count[:, None] - walk), count[:, None])
        out.append(value.min(axis=1) + len(x) - count)
    return np.concatenate(out).astype(np.int32)


def exact(case, seed):
    if case["call"] != "depth" or case["data"] == "int32" or case["algorithm"] != "rcom":
        return None
    n, p, m = case["n"], case["p"], case["m"]
    if p == 2 and n * m <= 4e7:
        return _flat(*_dataset(case, seed))
    if p == 3 and 0.5 * n ** 3 * m <= 1e9 and n >= 20:
        x, z = _dataset(case, seed)
        return np.array([_space(x, q) for q in z], dtype=np.int32)
    return None
