"""Plain FP64 form at p = 1, 2, 3, 4 (reciprocal steps and square roots) and
a general power against the FP64 oracle: tile edges, hits, points at infinity,
coordinates far outside FP32's range."""
import numpy as np
import pytest

import oracle
import synthetic

pytestmark = pytest.mark.gpu

TOL = 1e-13  # the FP64 form's bar, of the largest |z|


@pytest.mark.parametrize("p", [1.0, 2.0, 3.0, 4.0, 2.5])
@pytest.mark.parametrize("n,m,scale", [(1, 5, 1.0), (127, 1025, 1.0), (129, 64, 1e100),
                                       (1000, 1023, 1e-100), (5003, 333, 1.0)])
def test_parity(p, n, m, scale):
    import torch
    import paper_1402_4986_gb300 as idw
    prob = synthetic.uniform_problem(n, m, seed=n, exact_hits=min(n, 3))
    data, q = prob["data"].astype(np.float64), prob["queries"].astype(np.float64)
    Z64, _ = oracle.idw(data, q, p)
    if n > 1:
        data = np.concatenate([data, [[np.inf, 0.0, 5.0]]])  # weight 0
    data[:, :2] *= scale
    Z = idw.interpolate(torch.from_numpy(data).cuda(), torch.from_numpy(q * scale).cuda(), p, "f64")
    assert np.max(np.abs(Z.cpu().numpy() - Z64)) <= TOL * np.max(np.abs(prob["data"][:, 2]))
