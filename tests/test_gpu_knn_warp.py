"""The k-NN search by warps (few queries, or queries whose surroundings are
empty or dense) against the FP64 oracle: neighbour lists equal, k-th key and
hits equal, values within the FP32 bar.  Sizes sit at its edges: one and a
few points, fewer points than k, buffers of 32, 64 and more keys, ties, the
call sizes where the search changes, and queries outside the data's box."""
import numpy as np
import pytest

import oracle
import synthetic

pytestmark = pytest.mark.gpu


def _check(data, queries, k, p=2.0, index=False):
    import torch
    import paper_1402_4986_gb300 as idw
    d, q = torch.from_numpy(data).cuda(), torch.from_numpy(queries).cuda()
    if index:
        Z, nbr, kd2 = idw.LocalIndex(d, k=8).knn(q, p, k, neighbours=True, kth_d2=True)
    else:
        Z, nbr, kd2 = idw.interpolate_knn(d, q, p, k, neighbours=True, kth_d2=True)
    idw.sync_status()
    want = oracle.idw_knn(data, queries, p, k)
    assert np.array_equal(nbr.cpu().numpy(), want["nbr"])
    assert np.array_equal(kd2.cpu().numpy(), want["kd2"].astype(np.float32))
    err = np.abs(Z.cpu().numpy() - want["Z"])
    assert np.max(err) <= 2e-6 * np.max(np.abs(data[:, 2]))


@pytest.mark.parametrize("k", [1, 2, 8, 31, 32, 33, 63, 64])
@pytest.mark.parametrize("n", [1, 5, 64, 3001])
def test_few_queries(n, k):
    prob = synthetic.uniform_problem(n, 203, seed=n + k, exact_hits=min(n, 5))
    _check(prob["data"], prob["queries"], k, index=n > 64)


@pytest.mark.parametrize("k", [1, 8, 40])
def test_clustered(k):
    prob = synthetic.config_local(n=20000, m=2000, clustered=True)
    q = prob["queries"] * 3.0 - 1.0  # a third of the box inside the data's
    _check(prob["data"], np.ascontiguousarray(q), k, p=3.5)


def test_hard_queries_of_a_larger_call():
    """10,000 queries at k = 1 (above the all-warps size of 9216): the queries
    far from the blobs go to warps, those inside to threads."""
    prob = synthetic.config_local(n=30000, m=10000, clustered=True)
    _check(prob["data"], prob["queries"], 1)


def test_ties_and_duplicates():
    """A lattice (equal distances throughout) with every point doubled, and
    queries on its points and cell centres: ties go to the lower index."""
    xy = synthetic.grid_xy(24)
    xy = np.concatenate([xy, xy])
    data = synthetic.pack_xyz(xy, np.arange(len(xy), dtype=np.float32) / len(xy))
    queries = np.concatenate([xy[:100], synthetic.grid_xy(12)]).astype(np.float32)
    for k in (3, 32, 50):
        _check(data, np.ascontiguousarray(queries), k)


def test_far_queries():
    """Queries from 10 to 1e9 box widths away."""
    prob = synthetic.uniform_problem(4000, 12, seed=9)
    q = (prob["queries"] + np.float32(10.0) ** np.arange(1, 13)[:, None] % np.float32(1e9))
    _check(prob["data"], np.ascontiguousarray(q.astype(np.float32)), 8)


def _fastest(call, reps=5):
    """Microseconds of one call among `reps`, the best of five turns."""
    import torch
    start, stop = (torch.cuda.Event(enable_timing=True) for _ in range(2))
    best = float("inf")
    call()
    for _ in range(5):
        start.record()
        for _ in range(reps):
            call()
        stop.record()
        stop.synchronize()
        best = min(best, start.elapsed_time(stop) / reps * 1e3)
    return best


@pytest.mark.parametrize("distance", [1e-3, 0.05, 0.4, 3.0])
@pytest.mark.parametrize("k", [1, 8, 40])
def test_beyond_each_edge_and_corner(distance, k):
    prob = synthetic.uniform_problem(20000, 0, seed=k)
    r = np.random.default_rng(k)
    along = r.random(24, dtype=np.float32)
    lo, hi = np.full(24, -distance, np.float32), np.full(24, 1 + distance, np.float32)
    sides = [lo, along, hi]
    queries = np.concatenate([np.stack([x, y], 1) for x in sides for y in sides])
    _check(prob["data"], np.ascontiguousarray(queries), k)


def test_beyond_the_edge_takes_no_longer():
    """Queries up to a box width outside walk the part of their disc that
    reaches the data, about as many points as those inside walk (2 times as
    long a call; 28 times when the disc's count ignored the edge)."""
    import torch
    import paper_1402_4986_gb300 as idw
    prob = synthetic.uniform_problem(1 << 20, 10007, seed=3)
    index = idw.LocalIndex(torch.from_numpy(prob["data"]).cuda(), k=8)
    inside = torch.from_numpy(prob["queries"]).cuda()
    outside = torch.where(inside < 0.5, inside - 1.0, inside + 1.0)
    assert _fastest(lambda: index.knn(outside)) <= 8 * _fastest(lambda: index.knn(inside))


@pytest.mark.parametrize("k", [5, 32, 33, 64])
def test_more_ties_than_the_buffer_holds(k):
    """Eight places at one distance from the query, 60 points on each, and a
    few nearer: the tie is wider than any buffer of keys."""
    step = np.float32(0.25)
    ring = step * np.array([[3, 4], [4, 3], [-3, 4], [-4, 3], [3, -4], [4, -3], [-3, -4], [5, 0]],
                           np.float32)
    near = step * np.array([[1, 0], [0, 2], [2, 2]], np.float32)
    xy = np.concatenate([np.tile(ring, (60, 1)), near])
    data = synthetic.pack_xyz(xy, np.linspace(-1, 1, len(xy), dtype=np.float32))
    _check(data, np.zeros((33, 2), np.float32), k)
    _check(data, np.zeros((33, 2), np.float32), k, p=3.5, index=True)


@pytest.mark.parametrize("k", [1, 2, 8])
@pytest.mark.parametrize("m", [20480, 24577, 36864, 60000])
def test_clustered_queries(m, k):
    """Queries in the data's blobs: listed for warps up to a size (the first
    three are limits for k = 1, 2 and 8), then a thread each.  The same queries
    in calls of 8192 are all warps'."""
    import torch
    import paper_1402_4986_gb300 as idw
    r = np.random.default_rng(m)
    xy = synthetic.mixture_xy(r, 50000 + m).astype(np.float32)
    data = synthetic.pack_xyz(xy[:50000], r.standard_normal(50000).astype(np.float32))
    d, q = torch.from_numpy(data).cuda(), torch.from_numpy(np.ascontiguousarray(xy[50000:])).cuda()
    Z, nbr, kd2 = idw.interpolate_knn(d, q, 2.0, k, neighbours=True, kth_d2=True)
    for i in range(0, m, 8192):
        part = q[i:i + 8192].contiguous()
        Zp, nbrp, kd2p = idw.interpolate_knn(d, part, 2.0, k, neighbours=True, kth_d2=True)
        assert torch.equal(nbr[i:i + 8192], nbrp) and torch.equal(kd2[i:i + 8192], kd2p)
        assert float((Z[i:i + 8192] - Zp).abs().max()) <= 2e-6 * float(d[:, 2].abs().max())


def test_half_the_queries_take_no_longer():
    """Half a million queries in the blobs of a million points against twice as
    many (0.7 of their time; twice their time when each had a warp)."""
    import torch
    import paper_1402_4986_gb300 as idw
    n = 1 << 20
    xy = synthetic.mixture_xy(np.random.default_rng(3), 2 * n).astype(np.float32)
    data = synthetic.pack_xyz(xy[:n], xy[:n, 0])
    d, q = torch.from_numpy(data).cuda(), torch.from_numpy(np.ascontiguousarray(xy[n:])).cuda()
    half = q[:500000].contiguous()
    few = _fastest(lambda: idw.interpolate_knn(d, half, 2.0, 8))
    assert few <= 1.2 * _fastest(lambda: idw.interpolate_knn(d, q, 2.0, 8))
