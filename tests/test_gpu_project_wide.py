"""The projection kernels' count of entries near a bucket edge."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


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
