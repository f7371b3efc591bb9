"""Radius-form queries that a whole warp walks (many more candidates than
their neighbours have): values, counts and gradients against the FP64 oracle,
mixed in one warp with empty, hit and ordinary queries, at call sizes that
end inside a warp."""
import numpy as np
import pytest

import oracle
import synthetic

pytestmark = pytest.mark.gpu


def _problem(n, m):
    """A dense blob in a sparse square; queries inside, outside, far away and
    on data points (some of those duplicated)."""
    rng = np.random.default_rng(n + m)
    prob = synthetic.uniform_problem(n, m, seed=m)
    data, q = prob["data"], prob["queries"]
    data[: n // 2, :2] = 0.5 + 0.02 * rng.standard_normal((n // 2, 2))
    data[n // 2: n // 2 + 20] = data[:20]
    q[::3] = 0.5 + 0.02 * rng.standard_normal(q[::3].shape)
    q[::7] = data[rng.integers(0, n // 2, len(q[::7])), :2]
    q[5::11] += 9.0
    return np.ascontiguousarray(data), np.ascontiguousarray(q.astype(np.float32))


@pytest.mark.parametrize("modified", [False, True])
@pytest.mark.parametrize("n,m,radius", [(4000, 1, 0.1), (4000, 33, 0.05), (6001, 1000, 0.05),
                                        (300, 257, float("inf"))])
@pytest.mark.parametrize("p", [2.0, 3.5])
def test_values_counts_gradients(modified, n, m, radius, p):
    import torch
    import paper_1402_4986_gb300 as idw
    data, q = _problem(n, m)
    d, qd = torch.from_numpy(data).cuda(), torch.from_numpy(q).cuda()
    fwd = idw.interpolate_modified if modified else idw.interpolate_local
    Z, cnt = fwd(d, qd, p, radius, counts=True)
    Zo, _, cnto = (oracle.idw_modified if modified else oracle.idw_local)(data, q, p, radius)
    assert np.array_equal(cnt.cpu().numpy(), cnto)
    Z = Z.cpu().numpy()
    assert np.array_equal(np.isnan(Z), np.isnan(Zo))
    ok = ~np.isnan(Zo)
    assert not ok.any() or np.max(np.abs(Z[ok] - Zo[ok])) <= 2e-6 * np.max(np.abs(data[:, 2]))

    g = np.random.default_rng(1).standard_normal(m).astype(np.float32)
    got = idw.local_backward(d, qd, p, radius, torch.from_numpy(g).cuda(), modified=modified)
    want = (oracle.idw_modified_grad if modified else oracle.idw_local_grad)(data, q, p, radius, g)
    for a, name in zip(got, ("grad_z", "grad_xy", "grad_q", "grad_p")):
        a, b = a.cpu().numpy().astype(np.float64), np.asarray(want[name])
        scale = np.max(np.abs(b))
        # the bar of the adjoints: 1e-4 of the largest magnitude
        assert np.max(np.abs(a - b)) <= 1e-4 * scale, name
