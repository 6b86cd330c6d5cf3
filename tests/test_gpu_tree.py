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


@pytest.mark.parametrize("n", [1, 31, 1000, 32768, 32769 + 777])
@pytest.mark.parametrize("scale", [0.02, 1.0, 60.0, 400.0, 40000.0])
def test_entry_order_and_rows(orc, qwlib, cuda, n, scale):
    """The sorted arrays and the bitmaps for spans from one bucket to past the
    counting sort's 1,024 and the one- and two-byte id rows: entries grouped by
    bid, inside a bid in groups of eight ids of one bank cycling through the
    banks; bitmap answers equal to the level path's."""
    import torch
    rng = np.random.default_rng(n)
    d, m = 5, 3
    X = (rng.standard_normal((n, d)) * scale).astype(np.float32)
    A = rng.standard_normal((m, d)).astype(np.float32)
    b = (rng.random(m) * 4).astype(np.float32)
    index = qwlib.Index(*(torch.from_numpy(x).to(cuda) for x in (X, A, b)), w=4.0, v=30, l=2,
                        bitmaps=n * scale < 2e6)
    H = orc.hash(X, A, b, 4.0)
    o, span, eb, ei = index.export()
    assert np.array_equal(o, H.min(0)) and np.array_equal(span, H.max(0) - H.min(0))
    for i in range(m):
        bid = H[:, i] - o[i]
        for t0 in range(0, n, 32768):
            ids = np.arange(t0, min(n, t0 + 32768))
            bank = (ids >> 2) & 31
            key = bid[ids].astype(np.int64) * 32 + bank
            order = np.argsort(key, kind="stable")
            rank = np.empty(ids.size, np.int64)
            starts = np.r_[True, np.diff(key[order]) != 0]
            rank[order] = np.arange(ids.size) - np.maximum.accumulate(np.where(starts, np.arange(ids.size), 0))
            want = ids[np.lexsort((ids, bank, rank >> 3, bid[ids]))]
            assert np.array_equal(ei[i, t0:t0 + ids.size], want)
            assert np.array_equal(eb[i, t0:t0 + ids.size], bid[want])
    if n * scale < 2e6:
        Q = torch.from_numpy(X[rng.integers(0, n, size=7)]).to(cuda)
        one = index.candidates(Q, 1, path="levels")
        two = index.candidates(Q, 1, path="bitmap", loads="direct")
        assert all(torch.equal(x, y) for x, y in zip(one, two))
    index.free()
