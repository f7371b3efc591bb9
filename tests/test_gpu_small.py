"""Problems and batches that take the one-launch path (n <= 12288, at most 256
tiles of 128 queries, n m <= 100 2^20, p <= 4; at p = 2 not those of fewer than
1500 points and more than 192 tiles): parity with
the FP64 oracle at its edges (cluster slices, chunks, query tiles, the largest
sizes), hits, FP64 recomputations, saved outputs, NaN and infinities, scales,
and the sizes just outside it."""
import numpy as np
import pytest

import oracle
import synthetic

pytestmark = pytest.mark.gpu

TOL = 2e-6  # the FP32 form's bar, of the largest |z|


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("p", [1.0, 2.0, 3.0, 4.0, 2.5])
@pytest.mark.parametrize("n,m", [(1, 1), (7, 128), (8, 129), (63, 64), (511, 5), (513, 1000),
                                 (4095, 700), (4096, 4096), (4096, 4097), (12288, 130),
                                 (12289, 130), (5, 32768), (5, 32769), (12288, 1000)])
def test_parity(p, n, m):
    import paper_1402_4986_gb300 as idw
    prob = synthetic.uniform_problem(n, m, seed=n + m, exact_hits=min(n, m, 6))
    Z, s0, hit = idw.interpolate_saved(_dev(prob["data"]), _dev(prob["queries"]), p)
    Z64, hit64 = oracle.idw(prob["data"], prob["queries"], p)
    assert np.max(np.abs(Z.cpu().numpy() - Z64)) <= TOL * np.max(np.abs(prob["data"][:, 2]))
    hit = hit.cpu().numpy()
    assert np.array_equal(hit[hit >= 0], hit64[hit64 >= 0])
    on = hit64 < 0
    d = prob["queries"][on, None].astype(np.float64) - prob["data"][None, :, :2].astype(np.float64)
    # S0 carries the weights' relative errors, 2e-6 in all at p = 4.
    S0 = ((d ** 2).sum(-1) ** (-0.5 * p)).sum(1)
    assert np.allclose(s0.cpu().numpy()[on], S0, rtol=2e-6, atol=0.0)
    assert np.isinf(s0.cpu().numpy()[~on]).all()


@pytest.mark.parametrize("n,m", [(16, 24576), (16, 24577), (1499, 24577), (1500, 24577),
                                 (1499, 32768)])
def test_parity_of_a_second_wave(n, m):
    """Both sides of the limits for a single problem at p = 2."""
    test_parity(2.0, n, m)


@pytest.mark.parametrize("p,scale", [(2.0, 2.0 ** -60), (2.0, 2.0 ** 60), (64.0, 1.0), (0.1, 1.0)])
def test_scales_and_recomputed(p, scale):
    import paper_1402_4986_gb300 as idw
    prob = synthetic.uniform_problem(900, 500, seed=3)
    d, q = prob["data"].copy(), prob["queries"] * np.float32(scale)
    d[:, :2] *= np.float32(scale)
    z = idw.interpolate(_dev(d), _dev(q), p).cpu().numpy()
    Z64, _ = oracle.idw(prob["data"], prob["queries"], p)
    assert np.max(np.abs(z - Z64)) <= TOL * np.max(np.abs(d[:, 2]))


@pytest.mark.parametrize("p", [2.0, 3.0, 2.5])
def test_nan_and_infinity(p):
    import torch
    import paper_1402_4986_gb300 as idw
    prob = synthetic.uniform_problem(300, 300, seed=4)
    data, q = prob["data"].copy(), prob["queries"].copy()
    data[17, 0] = np.inf  # weight 0
    q[5, 1] = np.nan
    q[9, 0] = np.inf
    z = idw.interpolate(_dev(data), _dev(q), p)
    Z64, _ = oracle.idw(np.delete(data, 17, 0), prob["queries"], p)
    assert torch.isnan(z[[5, 9]]).all()
    z = np.delete(z.cpu().numpy(), [5, 9])
    assert np.max(np.abs(z - np.delete(Z64, [5, 9]))) <= TOL * np.max(np.abs(data[:, 2]))


def test_same_bits_and_capture():
    import torch
    import paper_1402_4986_gb300 as idw
    prob = synthetic.uniform_problem(1000, 1021, seed=6, exact_hits=3)
    d, q = _dev(prob["data"]), _dev(prob["queries"])
    z = idw.interpolate(d, q, 2.0)
    out = torch.empty_like(z)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        idw.interpolate(d, q, 2.0, out=out)
    out.zero_()
    g.replay()
    assert torch.equal(out, z)


@pytest.mark.parametrize("p", [2.0, 3.0, 2.5])
@pytest.mark.parametrize("sizes", [[(1, 1), (300, 128), (5, 129), (12288, 3), (64, 700)],
                                   [(40, 20)] * 256, [(40, 129)] * 129])
def test_batch(p, sizes):
    import paper_1402_4986_gb300 as idw
    probs = [synthetic.uniform_problem(n, m, seed=i, exact_hits=min(n, m, 2))
             for i, (n, m) in enumerate(sizes)]
    zs = idw.interpolate_batched([_dev(q["data"]) for q in probs],
                                 [_dev(q["queries"]) for q in probs], p)
    for z, q in zip(zs, probs):
        Z64, _ = oracle.idw(q["data"], q["queries"], p)
        assert np.max(np.abs(z.cpu().numpy() - Z64)) <= TOL * np.max(np.abs(q["data"][:, 2]))


@pytest.mark.parametrize("n,m", [(13000, 500), (30000, 2048), (30000, 2049), (30000, 5000)])
def test_combine_lanes(n, m):
    """Problems beyond the one-launch path whose queries have many pieces (one
    or two query tiles) and few."""
    import paper_1402_4986_gb300 as idw
    prob = synthetic.uniform_problem(n, m, seed=m, exact_hits=3)
    z = idw.interpolate(_dev(prob["data"]), _dev(prob["queries"]), 2.0).cpu().numpy()
    Z64, _ = oracle.idw(prob["data"], prob["queries"], 2.0)
    assert np.max(np.abs(z - Z64)) <= TOL * np.max(np.abs(prob["data"][:, 2]))


@pytest.mark.parametrize("n", [2048, 2049, 12288])
@pytest.mark.parametrize("repeat", range(3))
def test_all_hits_of_a_full_gpu(n, repeat):
    """Every query a hit, more clusters than the GPU holds at once."""
    import paper_1402_4986_gb300 as idw
    prob = synthetic.uniform_problem(n, 8192, seed=n + repeat)
    data = prob["data"]
    rng = np.random.default_rng(repeat)
    queries = np.ascontiguousarray(data[rng.integers(0, n, 8192), :2])
    Z, s0, hit = idw.interpolate_saved(_dev(data), _dev(queries), 2.0)
    Z64, hit64 = oracle.idw(data, queries, 2.0)
    assert np.array_equal(hit.cpu().numpy(), hit64)
    assert np.array_equal(Z.cpu().numpy(), Z64.astype(np.float32))
    assert np.isinf(s0.cpu().numpy()).all()
