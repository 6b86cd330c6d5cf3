"""The bitmap path's count forms against the level path: levels with few live
groups per query (quads of lanes), with many, and with many queries per group
(the table form), for projection counts around its rows of 16 and bucket counts
around 4, 8 and 16 per projection."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,c,scale", [(5, 2, 1.0), (16, 2, 6.0), (17, 3, 1.0), (40, 2, 2.0),
                                       (64, 2, 1.0), (127, 2, 1.0)])
@pytest.mark.parametrize("n,nq", [(32768, 700), (33500, 9000), (300, 40)])
def test_count_forms(qwlib, cuda, n, nq, m, c, scale):
    import torch
    g = torch.Generator(device=cuda).manual_seed(n + m)
    d = 12
    centres = torch.rand((6, d), generator=g, device=cuda) * 4 * scale
    lab = torch.randint(0, 6, (n,), generator=g, device=cuda)
    X = (centres[lab] + torch.randn((n, d), generator=g, device=cuda)).contiguous()
    far = torch.randn((nq, d), generator=g, device=cuda) * 0.3
    far[: nq // 10] *= 100  # queries whose buckets hold no data
    Q = (X[torch.randint(0, n, (nq,), generator=g, device=cuda)] + far).contiguous()
    A = torch.randn((m, d), generator=g, device=cuda)
    b = torch.rand((m,), generator=g, device=cuda)
    v = min(3000, n - 10)
    index = qwlib.Index(X, A, b, w=1.0, c=c, v=v, l=max(1, (2 * m) // 3), bitmaps=True)
    want = index.candidates(Q, 10, path="levels")
    for loads, graph in (("direct", False), ("direct", True), ("fused", True), ("tma", False)):
        got = index.candidates(Q, 10, path="bitmap", loads=loads, graph=graph)
        for x, y in zip(got, want):
            assert torch.equal(x, y)
    index.free()


@pytest.mark.parametrize("k,v", [(10, 500), (10, 4086)])
@pytest.mark.parametrize("graph", [False, True])
def test_long_lists(qwlib, cuda, k, v, graph):
    """Last levels of a few to 100,000 candidates (listed whole, or counted first
    and listed as far as they are kept), tie classes of a few ids and of
    thousands."""
    import torch
    g = torch.Generator(device=cuda).manual_seed(7)
    n, d, m = 100_000, 6, 12
    size = torch.tensor([35_000, 33_000, 20_000, 9_000, 2_900, 100], device=cuda)
    lab = torch.repeat_interleave(torch.arange(6, device=cuda), size)
    lab = lab[torch.randperm(n, generator=g, device=cuda)]
    centres = torch.randn((6, d), generator=g, device=cuda) * 30
    X = (centres[lab] + torch.randn((n, d), generator=g, device=cuda) * 0.5).contiguous()
    Q = X[torch.randint(0, n, (300,), generator=g, device=cuda)]
    Q = (Q + torch.randn(Q.shape, generator=g, device=cuda) * 0.2).contiguous()
    A = torch.randn((m, d), generator=g, device=cuda)
    b = torch.rand((m,), generator=g, device=cuda)
    index = qwlib.Index(X, A, b, w=1.0, c=2, v=v, l=9, bitmaps=True)
    want = index.candidates(Q, k, path="levels")
    assert (want[2][:, 2] > 32_768).any()
    got = index.candidates(Q, k, path="bitmap", loads="direct", graph=graph)
    for x, y in zip(got, want):
        assert torch.equal(x, y)
    index.free()
