"""The one-sweep adjoint (both sides wanted, p >= 1) against the same sums in
FP64 and against the two sweeps (one side at a time): edges of data units and
query tiles, hits, FP64-recomputed queries, several panels."""
import numpy as np
import pytest

import oracle
import synthetic

pytestmark = pytest.mark.gpu

TOL = 1e-4  # the adjoint's bar against the oracle, of each gradient's largest magnitude
# Against FP64 sums with the same saved Z and S0: a term's FP32 arithmetic and
# MUFU values are within about 20 units of 2^-24 and a sum of 10^4 of them
# adds less than that again, 3e-6 in all, of the largest magnitude.
SUM_TOL = 1e-5


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _rel(a, b):
    a, b = np.asarray(a, np.float64), np.asarray(b, np.float64)
    return np.max(np.abs(a - b)) / max(np.max(np.abs(b)), 1e-300)


def _sums64(prob, p, Z, s0, hit, g):
    """The adjoint's sums in FP64 from the forward pass's Z, S0 and hits."""
    x, z = prob["data"][:, :2].astype(np.float64), prob["data"][:, 2].astype(np.float64)
    on = hit == -1
    d = prob["queries"][on, None].astype(np.float64) - x[None]
    d2 = (d ** 2).sum(-1)
    w = d2 ** (-0.5 * p)
    c = (g[on] / s0[on])[:, None]
    e = z[None] - Z[on, None].astype(np.float64)
    b = (c * p * e * w / d2)[..., None] * d
    gz = (c * w).sum(0)
    np.add.at(gz, hit[hit >= 0], g[hit >= 0])
    gq = np.zeros((len(g), 2))
    gq[on] = -b.sum(1)
    return gz, b.sum(0), gq, float((-0.5 * c * e * w * np.log(d2)).sum())


@pytest.mark.parametrize("p", [1.0, 2.0, 2.5])
@pytest.mark.parametrize("n,m", [(1, 1), (2, 1023), (63, 1025), (65, 300), (127, 2049), (129, 4097),
                                 (3001, 2500), (20003, 77)])
def test_against_oracle_and_two_sweeps(p, n, m):
    import paper_1402_4986_gb300 as idw
    prob = synthetic.uniform_problem(n, m, seed=n + m, exact_hits=min(n, m, 3) if n > 1 else 0)
    d, q = _dev(prob["data"]), _dev(prob["queries"])
    gn = np.random.default_rng(m).standard_normal(m).astype(np.float32)
    g = _dev(gn)
    Z, s0, hit = idw.interpolate_saved(d, q, p)
    gz, gxy, gq, gp = idw.backward(d, q, p, Z, s0, hit, g)
    hits = hit.cpu().numpy()
    if (hits != -2).all():  # queries redone in FP64 have their own sums
        rz, rxy, rq, rp = _sums64(prob, p, Z.cpu().numpy(), s0.cpu().numpy(), hits, gn)
        assert _rel(gz.cpu().numpy(), rz) <= SUM_TOL
        if n > 1:  # with one point these are zero up to rounding
            assert _rel(gxy.cpu().numpy(), rxy) <= SUM_TOL
            assert _rel(gq.cpu().numpy(), rq) <= SUM_TOL
            assert abs(float(gp[0]) - rp) <= SUM_TOL * max(abs(rp), float(np.abs(gn).sum()))
    # The two sweeps, and repeated calls bit for bit (queries redone in FP64
    # add their data-side terms with atomics).
    hz, hxy, _, _ = idw.backward(d, q, p, Z, s0, hit, g, need_query_xy=False, need_p=False)
    _, _, hq, _ = idw.backward(d, q, p, Z, s0, hit, g, need_z=False, need_data_xy=False)
    scale = lambda t: max(float(t.abs().max()), 1e-30)
    assert float((gz - hz).abs().max()) <= 2 * SUM_TOL * scale(hz)
    assert n == 1 or float((gxy - hxy).abs().max()) <= 2 * SUM_TOL * scale(hxy)
    assert n == 1 or float((gq - hq).abs().max()) <= 2 * SUM_TOL * scale(hq)
    for a, b in zip(idw.backward(d, q, p, Z, s0, hit, g), (gz, gxy, gq, gp)):
        assert bool((a == b).all()) or (hits == -2).any()


def test_several_panels():
    """n = 2^20 points: a panel holds 21 tiles of 4096 queries; 90,000 queries
    make 22.  The data side of one and two panels agrees with one side alone."""
    import torch
    import paper_1402_4986_gb300 as idw
    torch.manual_seed(3)
    n, m = 1 << 20, 90000
    d = torch.rand(n, 3, device="cuda")
    q = torch.rand(m, 2, device="cuda")
    g = torch.randn(m, device="cuda")
    Z, s0, hit = idw.interpolate_saved(d, q, 2.0)
    gz, gxy, gq, _ = idw.backward(d, q, 2.0, Z, s0, hit, g, need_p=False)
    hz, hxy, _, _ = idw.backward(d, q, 2.0, Z, s0, hit, g, need_query_xy=False, need_p=False)
    _, _, hq, _ = idw.backward(d, q, 2.0, Z, s0, hit, g, need_z=False, need_data_xy=False,
                               need_p=False)
    for a, b in ((gz, hz), (gxy, hxy), (gq, hq)):
        assert float((a.double() - b).norm() / b.double().norm()) <= 1e-5


def test_extreme_pairs():
    """Pairs at 1e-18 of the extent (outside FP32's range of w / d^2 at p = 3)
    are redone in FP64; p below 1 takes the two sweeps."""
    import paper_1402_4986_gb300 as idw
    prob = synthetic.uniform_problem(700, 400, seed=5)
    prob["data"][:20, :2] = 0.0
    prob["data"][:20, 0] = np.arange(1, 21) * np.float32(1e-18)
    prob["queries"][:5] = 0.0
    prob["queries"][:5, 1] = np.arange(1, 6) * np.float32(3e-19)
    gn = np.ones(400, np.float32)
    for p in (3.0, 0.5):
        d, q = _dev(prob["data"]), _dev(prob["queries"])
        Z, s0, hit = idw.interpolate_saved(d, q, p)
        gz, gxy, gq, gp = idw.backward(d, q, p, Z, s0, hit, _dev(gn))
        G = oracle.idw_grad(prob["data"], prob["queries"], p, gn)
        assert _rel(gz.cpu().numpy(), G["grad_z"]) <= TOL
        assert _rel(gq.cpu().numpy(), G["grad_q"]) <= TOL


def test_without_room_for_the_partial_sums():
    """2^20 points want 252 MiB of them and 24 MiB of sums over panels, 403 MiB in
    all with the quarter that a handle adds; with 256 MiB of the device's memory
    left the two sweeps run, which need 86."""
    import torch
    import paper_1402_4986_gb300 as idw
    torch.manual_seed(4)
    n, m = 1 << 20, 90000
    d, q = torch.rand(n, 3, device="cuda"), torch.rand(m, 2, device="cuda")
    g = torch.randn(m, device="cuda")
    roomy, tight = idw.Handle(0), idw.Handle(0)
    Z, s0, hit = idw.interpolate_saved(d, q, 2.0, handle=roomy)
    want = idw.backward(d, q, 2.0, Z, s0, hit, g, handle=roomy)
    got = idw.backward(d[:1000].contiguous(), q, 2.0, Z, s0, hit, g, handle=tight)  # outputs' memory
    del got
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    held = torch.empty(free - (256 << 20), dtype=torch.uint8, device="cuda")
    try:
        got = idw.backward(d, q, 2.0, Z, s0, hit, g, handle=tight)
    finally:
        del held
        torch.cuda.empty_cache()
    for a, b in zip(got, want):
        assert float((a.double() - b).norm()) <= 1e-5 * float(b.double().norm())
