"""Performance cases: the calls a user of the package makes, over the range of sizes and options it
is used with.

Kinds of case (``kind``):
  global   ``interpolate``: all data points weigh in; p = 2 or another power, float32 with
           compensated sums or plain float64
  batched  ``interpolate_batched``: many independent uneven problems in one call
  adjoint  ``idw`` under autograd: forward and every gradient of the global form
  radius   ``interpolate_local`` / ``interpolate_modified``, or a prepared ``LocalIndex``
  radius_grad  ``idw_local`` / ``idw_modified`` under autograd
  knn      ``interpolate_knn``, or a prepared ``LocalIndex``
  knn_grad ``idw_knn`` under autograd

``exact`` restates each of them in plain torch float64.
"""
from __future__ import annotations

import math
import random

import torch

import paper_1402_4986_gb300 as idw

_DEV = "cuda"
_CLOUDS = ("uniform", "clustered")  # data positions


def listed():
    return [
        # A few hundred stations and a small set of prediction points: latency.
        dict(name="global small", kind="global", n=1000, m=1021, p=2.0, precision="f32c",
             cloud="uniform", hits=0),
        # An ordinary raster block from scattered data, odd sizes, some prediction points on a
        # station (cross-checks, rasters that pass through the stations).
        dict(name="global ragged", kind="global", n=100003, m=65537, p=2.0, precision="f32c",
             cloud="uniform", hits=16),
        # The headline workload of the benchmark: a million by a million.
        dict(name="global largest", kind="global", n=1 << 20, m=1 << 20, p=2.0, precision="f32c",
             cloud="uniform", hits=0),
        # The other power of the published experiments, at one of their sizes (50 x 1024).
        dict(name="global power 3", kind="global", n=51200, m=51200, p=3.0, precision="f32c",
             cloud="uniform", hits=0),
        # The double-precision form, for users who need its accuracy.
        dict(name="global double", kind="global", n=20000, m=10007, p=2.0, precision="f64",
             cloud="uniform", hits=0),
        # One call for many small uneven problems (tiles, time steps, folds).
        dict(name="batched small", kind="batched", count=64, lo=256, hi=8192, sizes=5, p=2.0),
        # A training step through the global form with a learned power.
        dict(name="adjoint", kind="adjoint", n=65536, m=65536, p=2.5, learn_p=True,
             cloud="uniform"),
        # The local form on a million points, about 32 members per query.
        dict(name="radius", kind="radius", n=1 << 20, m=1 << 20, members=32.0, p=2.0,
             modified=False, counts=False, prepared=False, cloud="uniform"),
        # A training step through modified Shepard on clustered data.
        dict(name="modified gradient", kind="radius_grad", n=200003, m=150001, members=16.0, p=2.0,
             modified=True, learn_p=False, cloud="clustered"),
        # Nearest-neighbour interpolation of a million queries.
        dict(name="nearest", kind="knn", n=1 << 20, m=1 << 20, k=32, p=2.0, lists=False,
             prepared=False, cloud="uniform"),
        # Serving: small query batches against one prepared index of clustered data, with the
        # neighbour lists.
        dict(name="nearest index", kind="knn", n=1 << 20, m=10007, k=8, p=2.0, lists=True,
             prepared=True, cloud="clustered"),
        # A training step through the nearest-neighbour form at its default k.
        dict(name="nearest gradient", kind="knn_grad", n=262144, m=262144, k=16, p=2.0,
             learn_p=False, cloud="uniform"),
    ]


def _size(rng, lo, hi):
    """A size spread over the logarithm of [lo, hi], odd ones among them."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _sizes(rng, lo, hi, pairs):
    """(n, m) in [lo, hi] with n m <= pairs."""
    n = _size(rng, lo, hi)
    return n, _size(rng, lo, max(lo, min(hi, pairs // n)))


def _power(rng):
    return rng.choice([2.0, 2.0, 2.0, 1.0, 1.5, 2.5, 3.0, 3.5, 4.0])


def draw(rng: random.Random):
    kind = rng.choice(["global", "global", "global", "batched", "adjoint", "radius", "radius",
                       "radius_grad", "knn", "knn", "knn_grad"])
    cloud = rng.choice(_CLOUDS)
    if kind == "global":
        precision = rng.choice(["f32c", "f32c", "f32c", "f64"])
        p = _power(rng)
        pairs = 1 << (32 if precision == "f64" else 38)
        if precision == "f64" and p != 2.0:
            pairs >>= 3
        n, m = _sizes(rng, 200, 1 << 20, pairs)
        return dict(kind=kind, n=n, m=m, p=p, precision=precision, cloud=cloud,
                    hits=rng.choice([0, 0, min(16, m // 64)]))
    if kind == "batched":
        hi = rng.choice([2048, 8192, 32768])
        return dict(kind=kind, count=rng.randint(2, 48), lo=256, hi=hi, sizes=rng.randrange(1000),
                    p=_power(rng))
    if kind == "adjoint":
        n, m = _sizes(rng, 500, 1 << 18, 1 << 35)
        return dict(kind=kind, n=n, m=m, p=_power(rng), learn_p=rng.random() < 0.5, cloud=cloud)
    if kind in ("radius", "radius_grad"):
        n, m = _size(rng, 1000, 1 << 20), _size(rng, 1000, 1 << 20)
        case = dict(kind=kind, n=n, m=m, members=float(rng.choice([4, 8, 16, 32, 64])),
                    p=_power(rng), modified=rng.random() < 0.5, cloud=cloud)
        if kind == "radius":
            case.update(counts=rng.random() < 0.5, prepared=rng.random() < 0.3)
        else:
            case.update(learn_p=rng.random() < 0.5)
        return case
    n, m = _size(rng, 1000, 1 << 20), _size(rng, 1000, 1 << 20)
    k = rng.choice([1, 3, 4, 8, 12, 16, 24, 32, 48, 64])
    case = dict(kind=kind, n=n, m=m, k=k, p=_power(rng), cloud=cloud)
    if kind == "knn":
        case.update(lists=rng.random() < 0.5, prepared=rng.random() < 0.4)
    else:
        case.update(learn_p=rng.random() < 0.5)
    return case


# ------------------------------------------------------------------ inputs


def _points(gen, n, cloud, dtype):
    """n data positions: uniform in the unit square, or 64 Gaussian blobs of sigma 0.01."""
    if cloud == "uniform":
        return torch.rand(n, 2, generator=gen, device=_DEV, dtype=dtype)
    centres = torch.rand(64, 2, generator=gen, device=_DEV, dtype=dtype)
    which = torch.randint(0, 64, (n,), generator=gen, device=_DEV)
    return centres[which] + 0.01 * torch.randn(n, 2, generator=gen, device=_DEV, dtype=dtype)


def _problem(gen, n, m, cloud="uniform", dtype=torch.float32, hits=0):
    """Data rows (x, y, z) of a smooth field with noise, and uniform queries."""
    xy = _points(gen, n, cloud, dtype)
    z = torch.sin(2 * math.pi * xy[:, 0]) * torch.cos(2 * math.pi * xy[:, 1])
    z += 0.1 * torch.randn(n, generator=gen, device=_DEV, dtype=dtype)
    data = torch.cat([xy, z[:, None]], 1).contiguous()
    queries = torch.rand(m, 2, generator=gen, device=_DEV, dtype=dtype)
    if hits:
        queries[torch.randperm(m, generator=gen, device=_DEV)[:hits]] = \
            xy[torch.randint(0, n, (hits,), generator=gen, device=_DEV)]
    return data, queries


def _radius(case):
    """R with ``members`` points within it at the unit square's mean density."""
    return math.sqrt(case["members"] / (math.pi * case["n"]))


def _batch_sizes(case):
    r = random.Random(case["sizes"])
    return [(_size(r, case["lo"], case["hi"]), _size(r, case["lo"], case["hi"]))
            for _ in range(case["count"])]


def _inputs(case, seed):
    gen = torch.Generator(device=_DEV)
    gen.manual_seed(int(seed))
    if case["kind"] == "batched":
        pairs = [_problem(gen, n, m) for n, m in _batch_sizes(case)]
        return {"datas": [d for d, _ in pairs], "queries": [q for _, q in pairs]}
    dtype = torch.float64 if case.get("precision") == "f64" else torch.float32
    data, queries = _problem(gen, case["n"], case["m"], case["cloud"], dtype, case.get("hits", 0))
    out = {"data": data, "queries": queries}
    if case["kind"] in ("adjoint", "radius_grad", "knn_grad"):
        out["g"] = torch.randn(case["m"], generator=gen, device=_DEV)
    return out


def prepare(case, seed):
    state = dict(_inputs(case, seed), case=case)
    if case.get("prepared"):
        state["index"] = (idw.LocalIndex(state["data"], k=case["k"]) if case["kind"] == "knn"
                          else idw.LocalIndex(state["data"], radius=_radius(case)))
    if "g" in state:  # the leaves of a training step
        state["data"].requires_grad_(True)
        state["queries"].requires_grad_(True)
        state["p"] = (torch.tensor(case["p"], device=_DEV, requires_grad=True)
                      if case["learn_p"] else case["p"])
    return state


def run(state):
    case = state["case"]
    kind, p = case["kind"], case.get("p")
    if kind == "global":
        return idw.interpolate(state["data"], state["queries"], p, precision=case["precision"])
    if kind == "batched":
        # One output for the whole batch, each problem writing its own part.
        sizes = [q.shape[0] for q in state["queries"]]
        out = torch.empty(sum(sizes), device=_DEV)
        idw.interpolate_batched(state["datas"], state["queries"], p, outs=list(out.split(sizes)))
        return out
    if kind == "radius":
        if case["prepared"]:
            return state["index"].interpolate(state["queries"], p, counts=case["counts"],
                                              modified=case["modified"])
        fn = idw.interpolate_modified if case["modified"] else idw.interpolate_local
        return fn(state["data"], state["queries"], p, _radius(case), counts=case["counts"])
    if kind == "knn":
        if case["prepared"]:
            return state["index"].knn(state["queries"], p, neighbours=case["lists"],
                                      kth_d2=case["lists"])
        return idw.interpolate_knn(state["data"], state["queries"], p, case["k"],
                                   neighbours=case["lists"], kth_d2=case["lists"])
    if kind == "adjoint":
        z = idw.idw(state["data"], state["queries"], state["p"])
    elif kind == "radius_grad":
        fn = idw.idw_modified if case["modified"] else idw.idw_local
        z = fn(state["data"], state["queries"], state["p"], _radius(case))
    else:
        z = idw.idw_knn(state["data"], state["queries"], state["p"], case["k"])
    leaves = [state["data"], state["queries"]] + ([state["p"]] if case["learn_p"] else [])
    return (z.detach(),) + torch.autograd.grad(z, leaves, state["g"])


# ------------------------------------------------------------- work, tolerance


def work(case):
    """Inputs read once, outputs written once; operations of the weighted pairs alone (a pair: two
    differences, d^2, a weight, two sums; a gradient pair about three times that)."""
    kind = case["kind"]
    per_pair = 9 if case.get("p") == 2.0 else 13
    if kind == "batched":
        sizes = _batch_sizes(case)
        return {"bytes": sum(12 * n + 12 * m for n, m in sizes),
                "flops": per_pair * sum(n * m for n, m in sizes)}
    n, m = case["n"], case["m"]
    word = 8 if case.get("precision") == "f64" else 4
    grad = kind in ("adjoint", "radius_grad", "knn_grad")
    size = word * (3 * n + 3 * m)
    if grad:  # upstream gradient in; data and query gradients out
        size += word * (m + 3 * n + 2 * m)
    if kind in ("global", "adjoint"):
        pairs = n * m
    elif kind in ("radius", "radius_grad"):
        pairs = m * case["members"]
        size += 4 * m if case.get("counts") else 0
    else:
        pairs = m * min(case["k"], n)
        size += 4 * m * (case["k"] + 1) if case.get("lists") else 0
    return {"bytes": size, "flops": per_pair * pairs * (4 if grad else 1)}


def tolerance(case):
    """About four times the difference from ``exact`` that was measured: 5e-8 for float32 values,
    4e-6 for float32 gradients (1e-3 of the root mean square for the worst single one, whose terms
    cancel), 5e-16 for float64 values.  Counts and neighbour lists are definite."""
    if case.get("precision") == "f64":
        return {"rel": 2e-15, "max": 1e-13}
    if case["kind"] in ("adjoint", "radius_grad", "knn_grad"):
        return {"rel": 1.6e-5, "max": 4e-3}
    return {"rel": 3e-7, "max": 2e-5, "differ": 0.0}


# ------------------------------------------------------------- float64 restatement


def _key32(q, x):
    """The FP32 squared distance that decides membership and nearness,
    fmaf(dy, dy, fl(dx dx)): every step is exact or rounded once in float64."""
    d = (q.float() - x.float()).double()
    t = (d[..., 0] * d[..., 0]).float().double()
    return (d[..., 1] * d[..., 1] + t).float()


def _chunks(m, width):
    step = max(1, (1 << 25) // max(1, width))
    for a in range(0, m, step):
        yield a, min(m, a + step)


def _in_reach(data, queries, reach):
    """Chunks (queries a..b, candidate indices, mask): for each query every data point within
    ``reach`` of it and more, from a grid of cells ``reach`` wide."""
    xy = data[:, :2].double()
    lo = xy.min(0).values
    cells = ((xy - lo) / reach).floor().long()
    gx, gy = (int(v) + 1 for v in cells.max(0).values)
    cell = cells[:, 1] * gx + cells[:, 0]
    order = torch.argsort(cell, stable=True)
    first = torch.searchsorted(cell[order], torch.arange(gx * gy + 1, device=_DEV))
    qc = ((queries.double() - lo) / reach).floor().long()
    rows = torch.stack([qc[:, 1] + d for d in (-1, 0, 1)], 1)
    x0, x1 = (qc[:, 0] - 1).clamp(0, gx), (qc[:, 0] + 2).clamp(0, gx)
    ok = (rows >= 0) & (rows < gy)
    base = rows.clamp(0, gy - 1) * gx
    start = torch.where(ok, first[base + x0[:, None]], 0)
    count = torch.where(ok, first[base + x1[:, None]], 0) - start
    end = count.cumsum(1)
    width = max(1, int(end[:, 2].max()))
    for a, b in _chunks(queries.shape[0], width):
        s = torch.arange(width, device=_DEV)[None, :]
        e = end[a:b]
        part = (s[..., None] >= e[:, None, :2]).sum(-1)
        before = torch.cat([torch.zeros_like(e[:, :1]), e[:, :2]], 1)
        at = torch.gather(start[a:b], 1, part) + s - torch.gather(before, 1, part)
        mask = s < e[:, 2:]
        yield a, b, order[torch.where(mask, at, 0)], mask


def _selection(case, data, queries):
    """Chunks (a, b, idx, member): each query's members under the local forms."""
    n, m = data.shape[0], queries.shape[0]
    if case["kind"] in ("radius", "radius_grad"):
        radius = _radius(case)
        r2 = torch.tensor(radius * radius, dtype=torch.float32, device=_DEV)
        for a, b, idx, mask in _in_reach(data, queries, radius * 1.0001):
            yield a, b, idx, mask & (_key32(queries[a:b, None], data[idx][..., :2]) < r2)
        return
    k = min(case["k"], n)
    top = torch.iinfo(torch.int64).max

    def nearest(q, idx, mask):
        d2 = _key32(q[:, None], data[idx][..., :2])
        key = (d2.view(torch.int32).long() << 32) | idx
        if mask is not None:
            key = torch.where(mask, key, top)
        return torch.topk(key, k, dim=1, largest=False, sorted=True).values

    keys = torch.full((m, k), top, device=_DEV)
    if case["cloud"] == "uniform" and n >= 4096:
        reach = 2.0 * math.sqrt(k / (math.pi * n)) + 1.0 / math.sqrt(n)
        for a, b, idx, mask in _in_reach(data, queries, reach):
            if idx.shape[1] >= k:
                got = nearest(queries[a:b], idx, mask)
                d2 = (got[:, -1] >> 32).int().view(torch.float32)
                keys[a:b] = torch.where(((got[:, -1] < top) & (d2 < (0.999 * reach) ** 2))[:, None],
                                        got, top)
    rest = (keys[:, -1] == top).nonzero()[:, 0]
    every = torch.arange(n, device=_DEV)[None, :]
    for a, b in _chunks(rest.shape[0], n):
        keys[rest[a:b]] = nearest(queries[rest[a:b]], every.expand(b - a, n), None)
    for a, b in _chunks(m, k):
        yield a, b, keys[a:b] & 0xffffffff, torch.ones(b - a, k, dtype=torch.bool, device=_DEV)


def _terms(q, x, member, p, radius):
    """Weights of the members (scaled by the heaviest), the factor f of dw/dq = -p f (q - x), and
    d ln w / dp; and the coincident members."""
    dx, dy = q[..., 0] - x[..., 0], q[..., 1] - x[..., 1]
    d2 = dx * dx + dy * dy
    hit = member & (d2 == 0)
    inf = float("inf")
    if radius is None:
        d2 = torch.where(member & (d2 > 0), d2, inf)
        s = d2.min(-1, keepdim=True).values
        r = torch.where(d2 < inf, s / d2, 0.0)
        w = r if p == 2.0 else r ** (0.5 * p)
        return dx, dy, w, w / d2, -0.5 * torch.log(torch.where(d2 < inf, d2 / s, 1.0)), hit
    d = torch.sqrt(torch.where(member & (d2 > 0), d2, inf))
    t = ((radius - d) / (radius * d)).nan_to_num(nan=0.0).clamp(min=0.0)
    s = t.max(-1, keepdim=True).values
    r = torch.where(s > 0, t / s, 0.0)
    w = r ** p
    on = t > 0
    f = torch.where(on, w / torch.where(on, t * d * d * d, 1.0), 0.0)
    return dx, dy, w, f, torch.where(on, torch.log(torch.where(on, r, 1.0)), 0.0), hit


def _value(w, z, idx, hit, none):
    """Z of a chunk: the weighted mean, the lowest coincident index's z, or NaN."""
    s0 = w.sum(-1)
    Z = (w * z).sum(-1) / s0
    big = torch.iinfo(torch.int64).max
    low = torch.where(hit, idx, big).min(-1)
    is_hit = low.values < big
    Z = torch.where(is_hit, torch.gather(z.expand_as(w), 1, low.indices[:, None])[:, 0], Z)
    return torch.where(none & ~is_hit, float("nan"), Z), s0, is_hit, low.values


def _exact_local(case, data, queries, g):
    n, m, p = data.shape[0], queries.shape[0], case["p"]
    radius = _radius(case) if case.get("modified") else None
    Z = torch.empty(m, dtype=torch.float64, device=_DEV)
    gd = torch.zeros(n, 3, dtype=torch.float64, device=_DEV)
    gq = torch.zeros(m, 2, dtype=torch.float64, device=_DEV)
    gp = torch.zeros((), dtype=torch.float64, device=_DEV)
    count = torch.empty(m, dtype=torch.int32, device=_DEV)
    rows = torch.empty(m, case.get("k", 0), dtype=torch.int32, device=_DEV)
    kd2 = torch.empty(m, device=_DEV)
    for a, b, idx, member in _selection(case, data, queries):
        x = data[idx].double()
        q = queries[a:b, None].double()
        dx, dy, w, f, lw, hit = _terms(q, x, member, p, radius)
        z = x[..., 2]
        Z[a:b], s0, is_hit, low = _value(w, z, idx, hit, ~member.any(-1))
        count[a:b] = torch.where(is_hit, -1, member.sum(-1)).int()
        if case.get("k"):
            rows[a:b] = idx.int()
            kd2[a:b] = _key32(queries[a:b], data[idx[:, -1], :2])
        if g is None:
            continue
        c = torch.where(is_hit | (s0 == 0), 0.0, g[a:b].double() / s0)[:, None]
        e = torch.where(c != 0, z - Z[a:b, None], 0.0)
        b2 = c * p * e * f
        terms = torch.stack([b2 * dx, b2 * dy, c * w], -1)
        gq[a:b] = -terms[..., :2].sum(1)
        gp += (c * e * w * lw).sum()
        gd.index_add_(0, idx.reshape(-1), terms.reshape(-1, 3))
        gd[:, 2].index_add_(0, low[is_hit], g[a:b][is_hit].double())
    return Z, gd, gq, gp, count, rows, kd2


def _exact_global(data, queries, p, g=None):
    n, m = data.shape[0], queries.shape[0]
    x = data.double()[None]
    z = x[..., 2]
    every = torch.arange(n, device=_DEV)[None, :]
    member = torch.ones(1, 1, dtype=torch.bool, device=_DEV)
    Z = torch.empty(m, dtype=torch.float64, device=_DEV)
    gd = torch.zeros(n, 3, dtype=torch.float64, device=_DEV)
    gq = torch.zeros(m, 2, dtype=torch.float64, device=_DEV)
    gp = torch.zeros((), dtype=torch.float64, device=_DEV)
    for a, b in _chunks(m, n):
        q = queries[a:b, None].double()
        if g is None:
            dx, dy = q[..., 0] - x[..., 0], q[..., 1] - x[..., 1]
            d2 = dx * dx + dy * dy
            s = torch.where(d2 > 0, d2, float("inf")).min(-1, keepdim=True).values
            hit = d2 == 0
            w = s / d2 if p == 2.0 else (s / d2) ** (0.5 * p)
            Z[a:b] = _value(w, z, every, hit, torch.zeros_like(hit[:, 0]))[0]
            continue
        dx, dy, w, f, lw, hit = _terms(q, x, member, p, None)
        Z[a:b], s0, is_hit, low = _value(w, z, every, hit, torch.zeros_like(hit[:, 0]))
        c = torch.where(is_hit, 0.0, g[a:b].double() / s0)[:, None]
        e = z - Z[a:b, None]
        b2 = c * p * e * f
        gx, gy = b2 * dx, b2 * dy
        gq[a:b] = -torch.stack([gx.sum(1), gy.sum(1)], 1)
        gp += (c * e * w * lw).sum()
        gd += torch.stack([gx.sum(0), gy.sum(0), (c * w).sum(0)], 1)
        gd[:, 2].index_add_(0, low[is_hit], g[a:b][is_hit].double())
    return Z, gd, gq, gp


def exact(case, seed):
    kind, p = case["kind"], case.get("p")
    pairs = (sum(n * m for n, m in _batch_sizes(case)) if kind == "batched"
             else case["n"] * case["m"])
    # Beyond these the restatement takes too long.
    limit = {"global": 3e10 if p == 2.0 else 6e9, "batched": 3e10 if p == 2.0 else 6e9,
             "adjoint": 5e9}.get(kind, 1e13 if case.get("cloud") == "uniform" or
                                 kind.startswith("radius") else 2.5e10)
    if pairs > limit:
        return None
    s = _inputs(case, seed)
    if kind == "batched":
        return torch.cat([_exact_global(d, q, p)[0] for d, q in zip(s["datas"], s["queries"])])
    if kind == "global":
        return _exact_global(s["data"], s["queries"], p)[0]
    if kind == "adjoint":
        Z, gd, gq, gp = _exact_global(s["data"], s["queries"], p, s["g"])
        return (Z, gd, gq) + ((gp,) if case["learn_p"] else ())
    Z, gd, gq, gp, count, rows, kd2 = _exact_local(case, s["data"], s["queries"], s.get("g"))
    if kind == "radius":
        return (Z, count) if case["counts"] else Z
    if kind == "knn":
        return (Z, rows, kd2.double()) if case["lists"] else Z
    return (Z, gd, gq) + ((gp,) if case["learn_p"] else ())
