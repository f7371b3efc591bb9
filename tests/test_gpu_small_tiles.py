"""Sizes for which the default rule picks the 512-query tiles: parity with
the FP64 oracle at their edges, single problems and batches."""
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
