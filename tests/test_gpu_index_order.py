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
