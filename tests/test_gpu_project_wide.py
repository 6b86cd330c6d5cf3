"""The projection kernels of larger blocks of vectors against the FP64 definition: the
switch from sums of pairs to the tiled kernel (256 rows), the 256-row tiles (blocks
of at least 100 tiles), and the number of entries near a bucket edge."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _vectors(n, d, m):
    rng = np.random.default_rng(n + 1000 * d + m)
    X = (rng.standard_normal((n, d)) * 4).astype(np.float32)
    X[::3] = rng.integers(-6, 7, size=X[::3].shape)
    X[n // 2] = 0.0
    X[-1] *= np.float32(1e4)
    A = rng.standard_normal((m, d)).astype(np.float32)
    A[::2] = rng.integers(-3, 4, size=A[::2].shape)
    b = (rng.random(m) * 4).astype(np.float32)
    b[::2] = np.floor(b[::2])
    return X, A, b


# rows: one side and the other of 256; of the line to the 256-row tiles (25,344 =
# 99 tiles; 12,544 and 12,801 with two column blocks); a last tile of 1 to 255
# rows; d and m off the multiples of four and of the column tiles of 32 and 64
@pytest.mark.parametrize("n,d,m", [(255, 9, 33), (256, 16, 64), (257, 17, 65), (25_344, 8, 33),
                                   (25_345, 12, 64), (25_347, 5, 31), (25_601, 7, 32),
                                   (12_544, 20, 65), (12_801, 17, 127), (40_001, 6, 100),
                                   (77_825, 7, 33), (77_827, 5, 31), (38_913, 17, 65)])
def test_hash_wide(orc, qwlib, cuda, n, d, m):
    import torch
    X, A, b = _vectors(n, d, m)
    H, fix = qwlib.hash(*(torch.from_numpy(x).to(cuda) for x in (X, A, b)), 4.0)
    assert np.array_equal(H.cpu().numpy(), orc.hash(X, A, b, 4.0))
    assert 0 <= fix <= H.numel()


@pytest.mark.parametrize("n,d,m", [(25_600, 12, 33), (25_603, 5, 20), (78_080, 6, 7),
                                   (50_050, 9, 65)])
def test_projection_major(orc, qwlib, cuda, n, d, m):
    """An index hashes its data projection by projection (whole 16-byte stores where
    the rows allow them): every entry's bucket as the definition gives it."""
    import torch
    X, A, b = _vectors(n, d, m)
    index = qwlib.Index(*(torch.from_numpy(x).to(cuda) for x in (X, A, b)), w=4.0, v=20, l=2)
    o, span, bid, ids = index.export()
    index.free()
    H = orc.hash(X, A, b, 4.0)
    assert np.array_equal(o, H.min(0)) and np.array_equal(span, H.max(0) - H.min(0))
    for i in range(m):
        assert np.array_equal(bid[i], H[ids[i], i] - o[i])


@pytest.mark.parametrize("n", [1, 100, 256, 257, 400])
def test_entries_near_an_edge(qwlib, cuda, n):
    """The count is of the entries within the first pass's bound B of an edge (or 1e-5,
    the larger), whichever kernel ran.  Integer products and offsets of 3e-6 buckets
    or of an eighth of one leave none between 1e-5 - B and 1e-5 + B, so the count is
    exact."""
    import torch
    rng = np.random.default_rng(n)
    d, m, w = 16, 24, 4.0
    X = rng.integers(-2, 3, size=(n, d)).astype(np.float32)
    A = rng.integers(-1, 2, size=(m, d)).astype(np.float32)
    b = np.where(np.arange(m) % 2, 0.5, 1.2e-5).astype(np.float32)
    u = (X.astype(np.float64) @ A.T.astype(np.float64) + b) / w
    near = np.abs(u - np.round(u))
    wt = np.arange(d, 0, -1.0)
    W = np.sqrt((X.astype(np.float64) ** 2) @ wt)[:, None] * np.sqrt((A.astype(np.float64) ** 2) @ wt)
    B = 2.0 ** -24 * (1.02 ** 3 * W / w + 4 * (np.abs(u) + 1))
    assert B.max() < 6e-6
    want = int((near <= 1e-5 - B).sum())
    assert want == int((near <= 1e-5 + B).sum()) and (n < 50 or want > n)
    fix = qwlib.hash(*(torch.from_numpy(x).to(cuda) for x in (X, A, b)), w)[1]
    assert fix == want


@pytest.mark.parametrize("tc", [False, True], ids=["fp32", "tensor"])
@pytest.mark.parametrize("offset", [1e3, 1e6])
@pytest.mark.parametrize("n,d,m", [(257, 33, 40), (300, 512, 64), (700, 16, 127), (2000, 24, 9),
                                   (9700, 8, 30)])
def test_hash_far_from_the_origin(orc, qwlib, cuda, n, d, m, offset, tc):
    """Rows whose first sums leave most entries open, in calls of few tiles (several
    blocks share a tile's entries)."""
    import torch
    rng = np.random.default_rng(n)
    X = (rng.standard_normal((n, d)) + offset).astype(np.float32)
    A = rng.standard_normal((m, d)).astype(np.float32)
    b = (rng.random(m) * 4).astype(np.float32)
    H, fix = qwlib.hash(*(torch.from_numpy(x).to(cuda) for x in (X, A, b)), 4.0, tensor_cores=tc)
    assert np.array_equal(H.cpu().numpy(), orc.hash(X, A, b, 4.0))
    assert 0 < fix <= H.numel() and (offset < 1e6 or fix > H.numel() * 0.9)
