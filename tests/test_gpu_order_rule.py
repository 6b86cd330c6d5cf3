"""QW_ORDER_AUTO: by signature from 2,048 queries on, or from 4e9 / n where that is
fewer; the results are those of the caller's order."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nq,ordered", [(5000, 2047, False), (5000, 2048, True),
                                          (2_100_000, 1904, False), (2_100_000, 1905, True)])
def test_order_auto(qwlib, cuda, n, nq, ordered):
    import torch
    g = torch.Generator(device=cuda).manual_seed(9)
    X = torch.randn((n, 6), generator=g, device=cuda)
    A = torch.randn((4, 6), generator=g, device=cuda)
    b = torch.rand((4,), generator=g, device=cuda)
    Q = X[torch.randint(0, n, (nq,), generator=g, device=cuda)].contiguous()
    index = qwlib.Index(X, A, b, w=0.2, v=30, l=3)
    want = index.query(Q, 3, stats=True, path="levels", order="given")
    index.profile(reset=True)
    got = index.query(Q, 3, stats=True, path="levels")
    assert (index.profile()["launches"]["order"] > 0) == ordered
    for x, y in zip(got, want):
        assert torch.equal(x, y)
    index.free()
