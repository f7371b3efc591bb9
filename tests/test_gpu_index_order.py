"""Query counts on both sides of the sizes up to which a prepared index leaves
its queries unsorted: the members, neighbour lists and values of the one-shot
calls (which sort), in the caller's query order."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [1, 255, 257, 1 << 17, (1 << 17) + 1])
def test_radius(m):
    import torch
    import paper_1402_4986_gb300 as idw
    torch.manual_seed(m)
    d, q = torch.rand(5000, 3, device="cuda"), torch.rand(m, 2, device="cuda")
    Z, cnt = idw.LocalIndex(d, radius=0.05).interpolate(q, 2.0, counts=True)
    Zo, cnto = idw.interpolate_local(d, q, 2.0, 0.05, counts=True)
    assert torch.equal(cnt, cnto)
    # The candidates' order may differ: last bits of z in [0, 1).
    assert float((Z - Zo).abs().max()) <= 2.0 ** -22


@pytest.mark.parametrize("m", [1 << 15, (1 << 15) + 1])
@pytest.mark.parametrize("k", [3, 40])
def test_knn(m, k):
    import torch
    import paper_1402_4986_gb300 as idw
    torch.manual_seed(m)
    d, q = torch.rand(5000, 3, device="cuda"), torch.rand(m, 2, device="cuda")
    Z, nbr = idw.LocalIndex(d, k=8).knn(q, 2.0, k, neighbours=True)
    Zo, nbro = idw.interpolate_knn(d, q, 2.0, k, neighbours=True)
    assert torch.equal(nbr, nbro)
    assert float((Z - Zo).abs().max()) <= 2.0 ** -22


@pytest.mark.parametrize("members", [20.0, 100.0, 700.0])
@pytest.mark.parametrize("m", [33, 20000, (1 << 17), (1 << 17) + 1])
def test_large_discs_in_any_order(m, members):
    """Up to 2^17 queries an index call leaves unsorted; those with many
    candidates are then warps'.  Against the one-shot call, which sorts."""
    import torch
    import paper_1402_4986_gb300 as idw
    import synthetic
    prob = synthetic.config_local(n=30000, m=m, members=members)
    d, q = torch.from_numpy(prob["data"]).cuda(), torch.from_numpy(prob["queries"]).cuda()
    Z, count = idw.LocalIndex(d, radius=prob["radius"]).interpolate(q, 2.0, counts=True)
    Zs, counts = idw.interpolate_local(d, q, 2.0, prob["radius"], counts=True)
    assert torch.equal(count, counts)
    assert torch.equal(Z.isnan(), Zs.isnan())
    assert float((Z - Zs).nan_to_num(0.0).abs().max()) <= 2e-6 * float(d[:, 2].abs().max())


def test_large_discs_take_no_longer_than_the_one_shot_call():
    """2^17 queries with 2048 members each: an index call, which saves the data's
    sort, against the one-shot call (level; 1.7 times as long when threads
    walked the unsorted queries' candidates)."""
    import torch
    import paper_1402_4986_gb300 as idw
    import synthetic
    from test_gpu_knn_warp import _fastest
    prob = synthetic.config_local(n=1 << 20, m=1 << 17, members=2048.0)
    d, q = torch.from_numpy(prob["data"]).cuda(), torch.from_numpy(prob["queries"]).cuda()
    index = idw.LocalIndex(d, radius=prob["radius"])
    once = _fastest(lambda: idw.interpolate_local(d, q, 2.0, prob["radius"]))
    assert _fastest(lambda: index.interpolate(q, 2.0)) <= 1.3 * once
