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


@pytest.mark.parametrize("p,ulps", [(1.0, 1.5), (2.0, 0.75), (3.0, 3.0), (4.0, 2.25)])
def test_weights(p, ulps):
    """S0 of one point is its weight.  Distances of 26 significant bits have
    exact squares of up to 52, whose low halves the hardware's approximation
    does not see; all exponents up to those where the weight leaves the normal
    range.  In ulps: a reciprocal 0.5 and the series' cut 2^-4, a square root's
    reciprocal 1 (its documented bound), and 0.5 for each product."""
    import torch
    import paper_1402_4986_gb300 as idw
    r = np.random.default_rng(64)
    top = int(1000 / max(p, 2.0))  # of the distance's exponent
    mant = r.integers(1 << 25, 1 << 26, 60000).astype(np.float64)
    mant[:4] = [1 << 25, (1 << 25) + 1, (1 << 26) - 1, (1 << 26) - 2]
    exp = r.integers(-top, top, mant.size)
    exp[:4] = [-top, top - 1, -top, top - 1]
    d = np.ldexp(mant, exp - 25)
    q = np.stack([d, np.zeros_like(d)], 1)
    data = torch.tensor([[0.0, 0.0, 1.0]], dtype=torch.float64, device="cuda")
    _, s0, hit = idw.interpolate_saved(data, torch.from_numpy(q).cuda(), p, "f64")
    assert (hit == -1).all()  # no value was redone
    # In 64 bits or more of the mantissa, whatever the machine's long double,
    # and of the mantissas alone: 2^(-p e) is exact.
    m = np.ldexp(mant, -25).astype(np.longdouble)
    want = {1.0: 1 / m, 2.0: 1 / (m * m), 3.0: 1 / (m * m) / m, 4.0: 1 / (m * m) / (m * m)}[p]
    got = np.ldexp(s0.cpu().numpy(), (p * exp).astype(int)).astype(np.longdouble)
    unit = np.spacing(want.astype(np.float64)).astype(np.longdouble)
    assert float(np.max(np.abs(got - want) / unit)) <= ulps
