"""The locality order at the edges of its nodes and chunks: an index with level
bitmaps answers as the oracle does whatever the shape of the tree."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _data(kind, n, d, rng):
    X = rng.standard_normal((n, d)).astype(np.float32) * 3
    if kind == "copies":        # every cut has all points on one side
        X[:] = X[0]
        X[-1] += 1
    elif kind == "ties":        # few distinct points: hyperplane distances tie
        X = X[rng.integers(0, min(5, n), size=n)]
    elif kind == "scales":      # one-sided cuts: each point far beyond the rest
        X *= (np.float32(1.07) ** (np.arange(n) % 120))[:, None].astype(np.float32)
    return np.ascontiguousarray(X, np.float32)


@pytest.mark.parametrize("kind", ["normal", "copies", "ties", "scales"])
@pytest.mark.parametrize("n,d,m", [(1, 3, 2), (128, 4, 3), (129, 5, 3), (256, 300, 4), (257, 64, 9),
                                   (385, 129, 5), (700, 3100, 3), (20_001, 6, 7)])
def test_tree_shapes(orc, qwlib, cuda, kind, n, d, m):
    import torch
    rng = np.random.default_rng(n + d)
    X = _data(kind, n, d, rng)
    Q = X[rng.integers(0, n, size=9)] + rng.standard_normal((9, d)).astype(np.float32) * 0.1
    A = rng.standard_normal((m, d)).astype(np.float32)
    b = (rng.random(m) * 4).astype(np.float32)
    k, v, l = min(3, n), 40, max(1, m // 2)
    w = float(4 * np.sqrt(d))
    H, HQ = orc.hash(X, A, b, w), orc.hash(Q, A, b, w)
    ref = orc.query(X, orc.build_index(H), Q, HQ, k=k, v=v, l=l, c=2)
    index = qwlib.Index(*(torch.from_numpy(x).to(cuda) for x in (X, A, b)), w=w, v=v, l=l,
                        bitmaps=True)
    ids, dists, st = index.query(torch.from_numpy(Q).to(cuda), k, stats=True, path="bitmap",
                                 loads="direct")
    assert np.array_equal(ids.cpu().numpy(), ref["ids"])
    assert np.array_equal(st.cpu().numpy(), ref["stats"])
    index.free()
