"""The bitmap path's table form with 8 and with 16 table rows per projection, where
nearly every group is live for every query, on both sides of the number of units that
the form asks for (2,000 queries with up to 32 projections make 96 of 200):
candidates, counts and statistics are the level path's."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,scale,rows", [(16, 1.2, 16), (33, 1.2, 16), (127, 0.5, 8), (20, 0.5, 8)])
@pytest.mark.parametrize("nq", [2000, 6000])
def test_table_rows(qwlib, cuda, m, scale, rows, nq):
    import torch
    n, d = 70_000, 12
    g = torch.Generator(device=cuda).manual_seed(m)
    X = torch.randn((n, d), generator=g, device=cuda) * scale
    A = torch.randn((m, d), generator=g, device=cuda)
    A = (A / A.norm(dim=1, keepdim=True)).contiguous()
    b = torch.rand((m,), generator=g, device=cuda)
    Q = (X[:nq] + torch.randn((nq, d), generator=g, device=cuda) * 0.05).contiguous()
    index = qwlib.Index(X, A, b, w=1.0, v=50, l=m // 2, bitmaps=True)
    assert rows // 2 <= index.info.span_max + 1 < rows
    want = index.candidates(Q, 10, path="levels")
    index.query(Q, 10, path="bitmap", loads="direct", profile=True)
    # the first level alone has the live groups that the form asks for
    later = int((want[2][:, 0] - 1).sum()) * ((n + 127) // 128)
    assert index.profile(reset=True)["bitmap_live_groups"] - later >= 256 * 256 * index.info.n_tiles
    for graph in (False, True):
        got = index.candidates(Q, 10, path="bitmap", loads="direct", graph=graph)
        for x, y in zip(got, want):
            assert torch.equal(x, y)
    index.free()
