"""The bitmap path where most groups are live and few queries run (data without
clusters, queries far from it): a task of four tiles is cut in parts over the grid's
warps; every level's counts and the candidates listed are the level path's."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("noise", [0.2, 8.0])
@pytest.mark.parametrize("v", [40, 1900, 4000])
@pytest.mark.parametrize("n,m", [(4000, 20), (70_001, 33), (300_000, 16)])
def test_parts(qwlib, cuda, n, m, v, noise):
    import torch
    g = torch.Generator(device=cuda).manual_seed(n + v)
    d = 24
    X = torch.randn((n, d), generator=g, device=cuda) * 3
    A = torch.randn((m, d), generator=g, device=cuda)
    b = torch.rand((m,), generator=g, device=cuda) * 4
    index = qwlib.Index(X, A, b, w=4.0, v=min(v, n - 10), l=(2 * m) // 3, bitmaps=True)
    for nq in (1, 2, 5, 17, 130, 400):
        Q = X[torch.randint(0, n, (nq,), generator=g, device=cuda)]
        Q = (Q + torch.randn(Q.shape, generator=g, device=cuda) * noise).contiguous()
        want = index.candidates(Q, 10, path="levels")
        for graph in (False, True):
            got = index.candidates(Q, 10, path="bitmap", loads="direct", graph=graph)
            for x, y in zip(got, want):
                assert torch.equal(x, y)
    index.free()
