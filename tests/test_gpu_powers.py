"""p = 1, 3 and 4 as powers of one reciprocal (square root): parity with the
FP64 oracle at the edges of chunks, tiles and query tiles, hits, batches,
points at infinity, NaN, and against the log2/exp2 form.  Calls with default
options lie within the one launch without a sweep; the tests that name a sweep
run the default sweep (512-query tiles) or a forced one at the same inputs."""
import numpy as np
import pytest

import oracle
import synthetic

pytestmark = pytest.mark.gpu

TOL = 2e-6  # the FP32 form's bar, of the largest |z|


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("p", [1.0, 3.0, 4.0])
@pytest.mark.parametrize("variant", [-1, 0, 4])
@pytest.mark.parametrize("n,m", [(1, 3), (31, 1), (32, 2049), (33, 4097), (257, 100), (5003, 777)])
def test_parity(p, variant, n, m):
    import paper_1402_4986_gb300 as idw
    h = idw.Handle(0)
    idw.set_option("sweep_variant", variant, handle=h)
    prob = synthetic.uniform_problem(n, m, seed=n + m, exact_hits=min(n, m, 4))
    Z, s0, hit = idw.interpolate_saved(_dev(prob["data"]), _dev(prob["queries"]), p, handle=h)
    Z64, hit64 = oracle.idw(prob["data"], prob["queries"], p)
    assert np.max(np.abs(Z.cpu().numpy() - Z64)) <= TOL * np.max(np.abs(prob["data"][:, 2]))
    hit = hit.cpu().numpy()
    assert np.array_equal(hit[hit >= 0], hit64[hit64 >= 0])
    on = hit64 < 0
    d = prob["queries"][on, None].astype(np.float64) - prob["data"][None, :, :2].astype(np.float64)
    # S0 carries the weights' relative errors: below p 2^-22 of the MUFU and
    # (p / 2 + 2) 2^-23 of the FP32 arithmetic, 2e-6 in all at p = 4.
    S0 = ((d ** 2).sum(-1) ** (-0.5 * p)).sum(1)
    assert np.allclose(s0.cpu().numpy()[on], S0, rtol=2e-6, atol=0.0)


@pytest.mark.parametrize("p", [1.0, 3.0, 4.0])
def test_batch_and_infinite_points(p):
    import torch
    import paper_1402_4986_gb300 as idw
    probs = [synthetic.uniform_problem(n, m, seed=n) for n, m in ((70, 300), (3000, 5000), (257, 9))]
    probs[1]["data"][5, 0] = np.inf  # weight 0
    outs = idw.interpolate_batched([_dev(q["data"]) for q in probs],
                                   [_dev(q["queries"]) for q in probs], p)
    for q, z in zip(probs, outs):
        d = q["data"][np.isfinite(q["data"]).all(1)]
        Z64, _ = oracle.idw(d, q["queries"], p)
        assert np.max(np.abs(z.cpu().numpy() - Z64)) <= TOL * np.max(np.abs(d[:, 2]))
    bad = probs[0]["queries"].copy()
    bad[7, 1] = np.nan
    z = idw.interpolate(_dev(probs[0]["data"]), _dev(bad), p)
    assert torch.isnan(z[7]) and torch.isfinite(z[:7]).all()


@pytest.mark.parametrize("p", [1.0, 3.0, 4.0])
@pytest.mark.parametrize("scale", [2.0 ** -60, 1.0, 2.0 ** 60])
def test_extreme_scales(p, scale):
    """Coordinates scaled by 2^+-60: the same weights up to the scale."""
    import paper_1402_4986_gb300 as idw
    prob = synthetic.uniform_problem(900, 500, seed=3)
    d, q = prob["data"].copy(), prob["queries"] * np.float32(scale)
    d[:, :2] *= np.float32(scale)
    z = idw.interpolate(_dev(d), _dev(q), p).cpu().numpy()
    Z64, _ = oracle.idw(prob["data"], prob["queries"], p)
    assert np.max(np.abs(z - Z64)) <= TOL * np.max(np.abs(d[:, 2]))


@pytest.mark.parametrize("p", [1.0, 3.0, 4.0])
@pytest.mark.parametrize("n,m", [(1, 3), (32, 2049), (33, 4097), (257, 100), (5003, 777)])
def test_parity_of_a_sweep(p, n, m, swept):
    import paper_1402_4986_gb300 as idw
    h = idw.Handle(0)
    prob = synthetic.uniform_problem(n, m, seed=n + m, exact_hits=min(n, m, 4))
    with swept(h):
        Z, s0, hit = idw.interpolate_saved(_dev(prob["data"]), _dev(prob["queries"]), p, handle=h)
    Z64, hit64 = oracle.idw(prob["data"], prob["queries"], p)
    assert np.max(np.abs(Z.cpu().numpy() - Z64)) <= TOL * np.max(np.abs(prob["data"][:, 2]))
    hit = hit.cpu().numpy()
    assert np.array_equal(hit[hit >= 0], hit64[hit64 >= 0])


@pytest.mark.parametrize("p", [1.0, 3.0, 4.0])
def test_batch_and_infinite_points_of_a_sweep(p, swept):
    with swept():
        test_batch_and_infinite_points(p)


@pytest.mark.parametrize("p", [1.0, 3.0, 4.0])
@pytest.mark.parametrize("variant", [-1, 0, 4])
@pytest.mark.parametrize("scale", [2.0 ** -60, 1.0, 2.0 ** 60])
def test_extreme_scales_of_a_sweep(p, scale, variant, swept):
    """Far padding (p = 4 shares reciprocals, p = 1 and 3 do not) against
    coordinates at both ends, a point at infinity among them."""
    import paper_1402_4986_gb300 as idw
    h = idw.Handle(0)
    idw.set_option("sweep_variant", variant, handle=h)
    prob = synthetic.uniform_problem(900, 500, seed=3)
    d, q = prob["data"].copy(), prob["queries"] * np.float32(scale)
    d[:, :2] *= np.float32(scale)
    d = np.concatenate([d, np.array([[np.inf, 0.0, 5.0]], np.float32)])  # weight 0
    with swept(h):
        z = idw.interpolate(_dev(d), _dev(q), p, handle=h).cpu().numpy()
    Z64, _ = oracle.idw(prob["data"], prob["queries"], p)
    assert np.max(np.abs(z - Z64)) <= TOL * np.max(np.abs(prob["data"][:, 2]))
