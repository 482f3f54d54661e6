"""The largest graphs that btas.apsp relaxes (n = 14400 fills a block's shared memory) and the first that go to blocked
Floyd-Warshall at once: the squarings' distances."""
import pytest

pytestmark = pytest.mark.gpu

INF = 0x3FFFFFFF


@pytest.mark.parametrize("n", [14400, 14401])
@pytest.mark.parametrize("w", [1000, 10 ** 6])
def test_sizes_around_the_limit(n, w):
    import torch

    import paper_1701_04733_gb300 as btas
    g = torch.Generator(device="cuda")
    g.manual_seed(n + w)
    W = torch.randint(1, w + 1, (n, n), dtype=torch.int32, device="cuda", generator=g)
    W.masked_fill_(torch.rand(n, n, device="cuda", generator=g) >= 8 / n, INF)
    W.fill_diagonal_(0)
    D, _ = btas.apsp(W, info=True)
    assert torch.equal(btas.apsp(W), D)
