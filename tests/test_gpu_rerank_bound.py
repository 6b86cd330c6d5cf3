"""The rerank's bound of the k-th smallest distance, against the oracle: distances
over thirty orders of magnitude (several refinements of a part), all equal, zero,
one far outlier, and candidate counts around the sizes of its count arrays."""
import numpy as np
import pytest

from test_gpu_parity import _full_parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,k", [(2, 1), (31, 30), (127, 5), (129, 128), (1000, 100), (4000, 7),
                                 (3900, 190)])
@pytest.mark.parametrize("kind", ["scales", "equal", "outlier"])
@pytest.mark.parametrize("rerank", ["fp32", "bf16", "bf16_tc"])
def test_bound(orc, qwlib, cuda, n, k, kind, rerank):
    rng = np.random.default_rng(n + k)
    d, m = 16, 4
    if kind == "scales":
        X = rng.standard_normal((n, d)) * 10.0 ** rng.uniform(-9, 6, size=(n, 1))
    elif kind == "equal":
        X = np.zeros((n, d))
        X[np.arange(n), rng.integers(0, d, size=n)] = 1.0
        X[: n // 3] = 0.0
    else:
        X = rng.standard_normal((n, d))
        X[n // 2] *= 1e12
    X = X.astype(np.float32)
    Q = np.concatenate([np.zeros((1, d)), X[:3] * 1.001, rng.standard_normal((2, d))])
    Q = np.ascontiguousarray(Q, np.float32)
    A = (rng.standard_normal((m, d)) * 1e-4).astype(np.float32)
    b = (rng.random(m) * 0.5).astype(np.float32)
    v = min(n, 4096 - k)
    _full_parity(orc, qwlib, cuda, X, Q, A, b, w=1.0, k=k, v=v, l=2, rerank=rerank)
