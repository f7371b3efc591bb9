"""Sizes for which the default rule picks the 512-query tiles: parity with
the FP64 oracle at their edges, single problems and batches.  (257, 300) and
test_batch lie within the one launch without a sweep; the tests that name a
sweep run the tiles there too."""
import numpy as np
import pytest

import oracle
import synthetic

pytestmark = pytest.mark.gpu

TOL = 2e-6  # the FP32 form's bar, of the largest |z|


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("p", [2.0, 3.0, 3.5])
@pytest.mark.parametrize("n,m", [(20000, 1), (20000, 512), (19999, 513), (40001, 2100), (257, 300)])
def test_single(p, n, m):
    import paper_1402_4986_gb300 as idw
    prob = synthetic.uniform_problem(n, m, seed=n + m, exact_hits=min(m, 3))
    h = idw.Handle(0)
    Z = idw.interpolate(_dev(prob["data"]), _dev(prob["queries"]), p, handle=h)
    # (257, 300) takes the one launch: the option then says what a sweep would be.
    if (p == 2.0 and n == 20000) or (p != 2.0 and n == 257):
        assert idw.get_option("last_variant", handle=h) in (6, 7)
    Z64, _ = oracle.idw(prob["data"], prob["queries"], p)
    assert np.max(np.abs(Z.cpu().numpy() - Z64)) <= TOL * np.max(np.abs(prob["data"][:, 2]))
    for v in (6, 7):  # picked by the rule only
        with pytest.raises(idw.IDWError):
            idw.set_option("sweep_variant", v, handle=h)


@pytest.mark.parametrize("p", [2.0, 3.0, 3.5])
def test_batch(p):
    import paper_1402_4986_gb300 as idw
    probs = [synthetic.uniform_problem(n, m, seed=n, exact_hits=1)
             for n, m in ((300, 511), (64, 513), (4097, 1), (1000, 1500), (256, 256)) * 6]
    outs = idw.interpolate_batched([_dev(q["data"]) for q in probs],
                                   [_dev(q["queries"]) for q in probs], p)
    for q, z in zip(probs, outs):
        Z64, _ = oracle.idw(q["data"], q["queries"], p)
        assert np.max(np.abs(z.cpu().numpy() - Z64)) <= TOL * np.max(np.abs(q["data"][:, 2]))


@pytest.mark.parametrize("p", [1.0, 2.0, 3.0, 3.5, 4.0])
@pytest.mark.parametrize("n,m,variants", [
    # work units of 64 points at p = 2 (6) and of 256 otherwise (7)
    (13000, 511, (6, 7)), (13000, 513, (6, 7)), (13000, 5000, (6, 7)), (30000, 4100, (7, 7)),
    (257, 300, (5, 7)), (20000, 1, (6, 7))])
def test_single_of_a_sweep(p, n, m, variants, swept):
    import paper_1402_4986_gb300 as idw
    prob = synthetic.uniform_problem(n, m, seed=n + m, exact_hits=min(m, 3))
    h = idw.Handle(0)
    with swept(h):
        Z = idw.interpolate(_dev(prob["data"]), _dev(prob["queries"]), p, handle=h)
    assert idw.get_option("last_variant", handle=h) == variants[p != 2.0]
    Z64, _ = oracle.idw(prob["data"], prob["queries"], p)
    assert np.max(np.abs(Z.cpu().numpy() - Z64)) <= TOL * np.max(np.abs(prob["data"][:, 2]))


def test_batch_of_a_sweep(swept):
    """The batch above at p = 2: 64-point units."""
    import paper_1402_4986_gb300 as idw
    with swept():
        test_batch(2.0)
    assert idw.get_option("last_variant") == 6


@pytest.mark.parametrize("p", [1.0, 3.0, 3.5, 4.0])
def test_large_batch(p):
    """64 problems of 256 to 8192, 3e8 pairs: above the one launch's limit, the
    256-point units of the 512-query tiles."""
    import paper_1402_4986_gb300 as idw
    r = np.random.default_rng(synthetic.DEFAULT_SEED)
    n, m = (np.exp(r.uniform(np.log(256), np.log(8192), 64)).astype(int) for _ in range(2))
    probs = [synthetic.uniform_problem(a, b, seed=a, exact_hits=1) for a, b in zip(n, m)]
    outs = idw.interpolate_batched([_dev(q["data"]) for q in probs],
                                   [_dev(q["queries"]) for q in probs], p)
    assert idw.get_option("last_variant") == 7
    for q, z in list(zip(probs, outs))[::7]:
        Z64, _ = oracle.idw(q["data"], q["queries"][::3], p)
        assert np.max(np.abs(z.cpu().numpy()[::3] - Z64)) <= TOL * np.max(np.abs(q["data"][:, 2]))
