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


@pytest.mark.parametrize("modified", [False, True])
def test_as_many_heavy_queries_as_fill_the_gpu(modified):
    """170,000 queries in the blobs of 20,000 points: most are heavy, so none is
    listed.  The same queries in calls of 85,000, which list theirs, give the
    same members, values and gradients."""
    import torch
    import paper_1402_4986_gb300 as idw
    m = 170000
    r = np.random.default_rng(5)
    xy = synthetic.mixture_xy(r, 20000 + m)
    data = synthetic.pack_xyz(xy[:20000], r.standard_normal(20000).astype(np.float32))
    d = torch.from_numpy(data).cuda()
    q = torch.from_numpy(np.ascontiguousarray(xy[20000:])).cuda()
    g = torch.from_numpy(r.standard_normal(m).astype(np.float32)).cuda()
    radius = synthetic.local_radius(20000, 16.0)
    call = idw.interpolate_modified if modified else idw.interpolate_local
    parts = [slice(0, m // 2), slice(m // 2, m)]
    Z, count = call(d, q, 2.5, radius, counts=True)
    gz, gxy, gq, gp = idw.local_backward(d, q, 2.5, radius, g, modified=modified)
    halves = [call(d, q[s].contiguous(), 2.5, radius, counts=True) for s in parts]
    grads = [idw.local_backward(d, q[s].contiguous(), 2.5, radius, g[s].contiguous(),
                                modified=modified) for s in parts]
    assert torch.equal(count, torch.cat([h[1] for h in halves]))
    Zh = torch.cat([h[0] for h in halves])
    assert torch.equal(Z.isnan(), Zh.isnan())
    assert float((Z - Zh).nan_to_num(0.0).abs().max()) <= 2e-6 * float(d[:, 2].abs().max())
    want = (grads[0][0] + grads[1][0], grads[0][1] + grads[1][1],
            torch.cat([grads[0][2], grads[1][2]]), grads[0][3] + grads[1][3])
    for a, b in zip((gz, gxy, gq, gp), want):
        # each within the adjoints' bar, 1e-4 of the largest magnitude
        assert float((a - b).abs().max()) <= 2e-4 * float(b.abs().max())
