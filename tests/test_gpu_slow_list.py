"""Flagged queries of large problems (exact hits, FP64 recomputations): listed
by the combine and finished by the two kernels after it, against the oracle.
Problems of up to 2048 points keep them in the combine; a list that is full
(more flagged queries than the staged tiles' memory holds records) leaves the
rest there too."""
import numpy as np
import pytest

import oracle
import synthetic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2048, 2049, 8193, 20011])
@pytest.mark.parametrize("m,p", [(33, 2.0), (700, 3.5), (20000, 2.0)])
def test_hits(n, m, p):
    """Every query on a data point, half of the points duplicated (the lowest
    index wins); 20000 hits overflow the list of 2049 and of 8193 points (1046 and 4886 records)."""
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
