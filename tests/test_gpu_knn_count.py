"""The k-NN search by counts (calls without neighbour lists on evenly spread
data: k > 32 above the all-warps size, k > 16 above 114,688 queries) and its
neighbours, against the list-returning searches of the same call and the FP64
oracle: k-th keys equal, values within the last bits, hits, ties, edges of the
data, clusters, fewer points than k, queries outside the box."""
import numpy as np
import pytest

import oracle
import synthetic

pytestmark = pytest.mark.gpu


def _compare(data, queries, k, p=2.0):
    import torch
    import paper_1402_4986_gb300 as idw
    d, q = torch.from_numpy(data).cuda(), torch.from_numpy(np.ascontiguousarray(queries)).cuda()
    Z, kd2 = idw.interpolate_knn(d, q, p, k, kth_d2=True)
    Zl, _, kd2l = idw.interpolate_knn(d, q, p, k, neighbours=True, kth_d2=True)
    idw.sync_status()
    assert torch.equal(kd2.nan_to_num(-1.0), kd2l.nan_to_num(-1.0))
    assert torch.equal(Z.isnan(), Zl.isnan())
    top = float(np.max(np.abs(data[:, 2])))
    # Both are correctly weighted sums of the same keys, within the FP32 bar.
    assert float((Z - Zl).nan_to_num(0.0).abs().max()) <= 2e-6 * top
    return Z.cpu().numpy()


@pytest.mark.parametrize("k", [1, 16, 17, 31, 32, 33, 64])
@pytest.mark.parametrize("n", [200, 5000, 60000])
def test_uniform(n, k):
    m = 8192 + 1024 * k + 1  # threads' (counted if k > 32), ending inside a warp
    prob = synthetic.uniform_problem(n, m, seed=n + k, exact_hits=100)
    Z = _compare(prob["data"], prob["queries"], k)
    part = slice(0, None, 97)
    want = oracle.idw_knn(prob["data"], prob["queries"][part], 2.0, k)["Z"]
    assert np.max(np.abs(Z[part] - want)) <= 2e-6 * np.max(np.abs(prob["data"][:, 2]))


@pytest.mark.parametrize("k", [8, 17, 40])
def test_clustered_and_outside(k):
    prob = synthetic.config_local(n=30000, m=50000, clustered=True)
    _compare(prob["data"], prob["queries"] * 2.0 - 0.5, k, p=3.5)


def test_ties():
    """A doubled lattice: bins of many equal keys, settled by index."""
    xy = synthetic.grid_xy(64)
    xy = np.concatenate([xy, xy])
    data = synthetic.pack_xyz(xy, np.arange(len(xy), dtype=np.float32) / len(xy))
    queries = np.tile(np.concatenate([xy[:4096], synthetic.grid_xy(32)]), (8, 1))
    for k in (5, 17, 30):
        _compare(data, queries.astype(np.float32), k)


def test_few_points_and_bad_queries():
    prob = synthetic.uniform_problem(5, 40000, seed=2)
    prob["queries"][7] = np.nan
    prob["queries"][8, 0] = np.inf
    Z = _compare(prob["data"], prob["queries"], 17)
    assert np.isnan(Z[7]) and np.isnan(Z[8]) and np.isfinite(Z[9:]).all()


@pytest.mark.parametrize("clustered", [False, True])
def test_largest_calls(clustered):
    """Above 2^19 queries clustered data are searched by heaps alone."""
    prob = synthetic.config_local(n=100000, m=(1 << 19) + 33, clustered=clustered)
    _compare(prob["data"], prob["queries"], 18)


@pytest.mark.parametrize("scale", [1e-15, 1e-30, 1e15])
def test_scales(scale):
    prob = synthetic.uniform_problem(3000, 40000, seed=4)
    prob["data"][:, :2] *= np.float32(scale)
    _compare(prob["data"], prob["queries"] * np.float32(scale), 20)


def test_up_to_32_neighbours_counted_from_114689_queries():
    """k = 17 .. 32 are counted above 7 * 2^14 queries."""
    m = 7 * (1 << 14) + 1
    for k in (17, 24, 32):
        prob = synthetic.uniform_problem(6000, m, seed=k, exact_hits=100)
        Z = _compare(prob["data"], prob["queries"], k)
        part = slice(0, None, 997)
        want = oracle.idw_knn(prob["data"], prob["queries"][part], 2.0, k)["Z"]
        assert np.max(np.abs(Z[part] - want)) <= 2e-6 * np.max(np.abs(prob["data"][:, 2]))


@pytest.mark.parametrize("share", [0.3, 0.45, 0.7])
def test_queries_beyond_the_edge(share):
    """120,000 queries, k = 20, a share of them beyond the data: the counting
    search leaves them to warps (36,000), to threads (54,000), or, where they
    are most of the call, does not run."""
    prob = synthetic.uniform_problem(5000, 120000, seed=8)
    q = prob["queries"]
    out = np.random.default_rng(8).random(len(q)) < share
    q[out] = np.where(q[out] < 0.5, q[out] - 0.7, q[out] + 0.7)
    Z = _compare(prob["data"], q, 20)
    part = slice(0, None, 499)
    want = oracle.idw_knn(prob["data"], np.ascontiguousarray(q[part]), 2.0, 20)["Z"]
    assert np.max(np.abs(Z[part] - want)) <= 2e-6 * np.max(np.abs(prob["data"][:, 2]))


def test_uneven_rims():
    """Data in a disc: even by the count of filled cells, with a fifth of the
    box empty; its queries are left over from the counting search."""
    prob = synthetic.uniform_problem(40000, 300000, seed=9)
    xy = prob["data"][:, :2]
    data = np.ascontiguousarray(prob["data"][((xy - 0.5) ** 2).sum(1) < 0.25])
    _compare(data, prob["queries"], 24)


@pytest.mark.parametrize("m", [1 << 18, (1 << 18) + 1, 1 << 19])
@pytest.mark.parametrize("clustered", [False, True])
def test_where_the_heap_search_is_started_another_way(m, clustered):
    prob = synthetic.config_local(n=20000, m=m, clustered=clustered)
    _compare(prob["data"], prob["queries"], 18)


def test_queries_beyond_the_edge_take_no_longer():
    """131,072 queries, most of them beyond the data, k = 32: without lists (the
    call that may count) against with lists (which never does).  About equal;
    11 times as long when every such query ended up with a warp of its own."""
    import torch
    import paper_1402_4986_gb300 as idw
    from test_gpu_knn_warp import _fastest
    prob = synthetic.uniform_problem(1 << 20, 1 << 17, seed=3)
    d = torch.from_numpy(prob["data"]).cuda()
    q = torch.from_numpy(prob["queries"]).cuda() * 3.0 - 1.0
    counted = _fastest(lambda: idw.interpolate_knn(d, q, 2.0, 32))
    assert counted <= 3 * _fastest(lambda: idw.interpolate_knn(d, q, 2.0, 32, neighbours=True))


def test_counted_ties():
    """As test_ties, with k and m that are counted: bins overflow on the ties."""
    xy = synthetic.grid_xy(64)
    xy = np.concatenate([xy, xy])
    data = synthetic.pack_xyz(xy, np.arange(len(xy), dtype=np.float32) / len(xy))
    queries = np.tile(np.concatenate([xy[:4096], synthetic.grid_xy(32)]), (24, 1))
    for k in (17, 30, 40):
        _compare(data, queries.astype(np.float32), k)


def test_counted_few_points_and_bad_queries():
    prob = synthetic.uniform_problem(5, 120000, seed=2)
    prob["queries"][7] = np.nan
    prob["queries"][8, 0] = np.inf
    for k in (17, 40):
        Z = _compare(prob["data"], prob["queries"], k)
        assert np.isnan(Z[7]) and np.isnan(Z[8]) and np.isfinite(Z[9:]).all()


@pytest.mark.parametrize("scale", [1e-15, 1e-30, 1e15])
def test_counted_scales(scale):
    prob = synthetic.uniform_problem(3000, 120000, seed=4)
    prob["data"][:, :2] *= np.float32(scale)
    for k in (20, 40):
        _compare(prob["data"], prob["queries"] * np.float32(scale), k)
