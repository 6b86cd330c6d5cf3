"""The projection kernels at the edges of their tiles, against the FP64 definition."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tc", [False, True], ids=["fp32", "tensor"])
@pytest.mark.parametrize("n,d,m", [(1, 1, 1), (3, 8, 33), (128, 17, 65), (1024, 31, 32),
                                   (1025, 33, 32), (1025, 7, 33), (1153, 64, 64), (1280, 16, 65),
                                   (2049, 100, 127)])
def test_hash_tile_edges(orc, qwlib, cuda, n, d, m, tc):
    """Rows and projections around the few-rows limit (1,024), the 128-row and
    32- and 64-projection tiles and the 16-coordinate chunk; a third of the rows
    are small integers (with b and w whole, those lie on bucket edges for integer
    projections, so pass 2 and its FP64 sequence decide), one row is zero and one
    is huge."""
    import torch
    rng = np.random.default_rng(n * 1000 + d)
    X = (rng.standard_normal((n, d)) * 4).astype(np.float32)
    X[::3] = rng.integers(-6, 7, size=X[::3].shape)
    X[n // 2] = 0.0
    X[-1] *= np.float32(1e4)
    A = rng.standard_normal((m, d)).astype(np.float32)
    A[::2] = rng.integers(-3, 4, size=A[::2].shape)
    b = (rng.random(m) * 4).astype(np.float32)
    b[::2] = np.floor(b[::2])
    want = orc.hash(X, A, b, 4.0)
    H, fix = qwlib.hash(*(torch.from_numpy(x).to(cuda) for x in (X, A, b)), 4.0, tensor_cores=tc)
    assert np.array_equal(H.cpu().numpy(), want)
    assert 0 <= fix <= want.size


@pytest.mark.parametrize("rows", [[0], [3, 40, 41], list(range(70))])
@pytest.mark.parametrize("n,d", [(70, 512), (70, 33), (300, 513)])
def test_entries_on_an_edge(orc, qwlib, cuda, n, d, rows):
    """Rows of integers whose projections fall exactly on a bucket's edge (summed
    in FP64 by a warp, or side by side, and then in the definition's order), among
    rows that the first sums decide."""
    import torch
    rng = np.random.default_rng(d)
    m = 9
    V = rng.standard_normal((n, d)).astype(np.float32)
    V[rows] = rng.integers(-3, 4, size=(len(rows), d))
    A = rng.integers(-2, 3, size=(m, d)).astype(np.float32)
    b = np.zeros(m, np.float32)
    got, _ = qwlib.hash(*(torch.from_numpy(x).to(cuda) for x in (V, A, b)), 1.0)
    assert np.array_equal(got.cpu().numpy(), orc.hash(V, A, b, 1.0))
