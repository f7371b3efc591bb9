"""Flagged queries of large problems (exact hits, FP64 recomputations): listed
by the combine and finished by the kernel after it, against the oracle.
Problems of up to 2048 points keep them in the combine; a list that is full
(more flagged queries than the staged tiles' memory holds records) leaves the
rest there too.  Calls within the limits of the one launch without a sweep (up
to 12,288 points and 100 * 2^20 pairs) finish their own: the tests that name a
sweep ask for one."""
import numpy as np
import pytest

import oracle
import synthetic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2048, 2049, 8193, 20011])
@pytest.mark.parametrize("m,p", [(33, 2.0), (700, 3.5), (20000, 2.0)])
def test_hits(n, m, p):
    """Every query on a data point, half of the points duplicated (the lowest
    index wins).  By default only 20,011 points and 20,000 queries on 8193 reach
    the list, which the latter overflow (4795 records); the rest take the one
    launch."""
    import torch
    import paper_1402_4986_gb300 as idw
    prob = synthetic.uniform_problem(n, m, seed=n + m)
    rng = np.random.default_rng(5)
    data = prob["data"]
    data[n // 2:, :2] = data[rng.integers(0, n // 2, n - n // 2), :2]
    queries = np.ascontiguousarray(data[rng.integers(0, n, m), :2])
    Z64, hit64 = oracle.idw(data, queries, p)
    Z, s0, hit = idw.interpolate_saved(torch.from_numpy(data).cuda(),
                                       torch.from_numpy(queries).cuda(), p)
    assert np.array_equal(hit.cpu().numpy(), hit64)
    assert np.array_equal(Z.cpu().numpy(), Z64.astype(np.float32))
    assert np.isinf(s0.cpu().numpy()).all()


def test_mixed_batch():
    """A batch whose flagged queries belong to several problems, small and
    large; at p = 64 the queries without a hit are recomputed in FP64."""
    import torch
    import paper_1402_4986_gb300 as idw
    probs = [synthetic.uniform_problem(n, m, seed=n, exact_hits=h)
             for n, m, h in ((9000, 50, 40), (500, 60, 10), (2049, 300, 7), (30000, 40, 40))]
    for p in (2.0, 64.0):
        outs = idw.interpolate_batched([torch.from_numpy(q["data"]).cuda() for q in probs],
                                       [torch.from_numpy(q["queries"]).cuda() for q in probs], p)
        for q, z in zip(probs, outs):
            Z64, hit64 = oracle.idw(q["data"], q["queries"], p)
            z = z.cpu().numpy()
            on = hit64 >= 0
            assert np.array_equal(z[on], Z64[on].astype(np.float32))
            # the bar of the FP32 form; FP64 results carry only their rounding
            assert np.max(np.abs(z - Z64)) <= 2e-6 * np.max(np.abs(q["data"][:, 2]))


@pytest.mark.parametrize("n", [2048, 2049, 8193, 20011])
@pytest.mark.parametrize("m,p", [(1, 2.0), (33, 2.0), (257, 1.0), (700, 3.5), (20000, 2.0)])
def test_hits_of_a_sweep(n, m, p, swept):
    """As test_hits, by the sweep at every size: the combine alone up to 2048
    points, then the list, whose kernel cuts few queries' points into many
    slices and draws many groups of queries one by one; 20,000 hits overflow
    the lists of 2049 and 8193 points."""
    with swept():
        test_hits(n, m, p)


def test_mixed_batch_of_a_sweep(swept):
    with swept():
        test_mixed_batch()


@pytest.mark.parametrize("hits", [0, 1, 300, 4000])
def test_hits_among_others_of_a_sweep(hits, swept):
    """Lists of no entry, of one, of more than a block's threads and of several
    rounds; the neighbours of a hit, whose sums it spoils, are on them too."""
    import torch
    import paper_1402_4986_gb300 as idw
    prob = synthetic.uniform_problem(30011, 8000, seed=hits, exact_hits=hits)
    Z64, hit64 = oracle.idw(prob["data"], prob["queries"], 2.0)
    d, q = torch.from_numpy(prob["data"]).cuda(), torch.from_numpy(prob["queries"]).cuda()
    with swept():
        for _ in range(2):  # the counts start over with each call
            Z, _, hit = idw.interpolate_saved(d, q, 2.0)
            on = hit64 >= 0
            assert np.array_equal(hit.cpu().numpy()[on], hit64[on])
            assert not (hit.cpu().numpy()[~on] >= 0).any()
            Zc = Z.cpu().numpy()
            assert np.array_equal(Zc[on], Z64[on].astype(np.float32))
            assert np.max(np.abs(Zc - Z64)) <= 2e-6 * np.max(np.abs(prob["data"][:, 2]))


@pytest.mark.parametrize("n,hits", [(300, 40), (2048, 40), (2048, 900), (2049, 2049), (8193, 8000)])
def test_hits_among_others_kept_by_the_combine(n, hits, swept):
    """As test_hits_among_others_of_a_sweep, where the combine's CTAs find the
    hits and sum the others in FP64: small problems, and lists that overflow."""
    import torch
    import paper_1402_4986_gb300 as idw
    prob = synthetic.uniform_problem(n, 20000, seed=n, exact_hits=hits)
    Z64, hit64 = oracle.idw(prob["data"], prob["queries"], 2.0)
    d, q = torch.from_numpy(prob["data"]).cuda(), torch.from_numpy(prob["queries"]).cuda()
    with swept():
        Z, _, hit = idw.interpolate_saved(d, q, 2.0)
    Z, hit, on = Z.cpu().numpy(), hit.cpu().numpy(), hit64 >= 0
    assert np.array_equal(hit[on], hit64[on])
    assert not (hit[~on] >= 0).any()
    assert np.array_equal(Z[on], Z64[on].astype(np.float32))
    assert np.max(np.abs(Z - Z64)) <= 2e-6 * np.max(np.abs(prob["data"][:, 2]))
