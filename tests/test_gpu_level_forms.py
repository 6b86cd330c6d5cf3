"""The level path at the edges of its parts, against the oracle: runs shorter
than one 8-id chunk, runs that start and end inside chunks, tiles of one id and
of all, one projection and the most, ties that fill a tile at the cut; and the
few-row form of the QALSH projection at its row, projection and coordinate
remainders."""
import numpy as np
import pytest

from test_gpu_parity import TILE, _full_parity
from test_gpu_qalsh import _parity as _qalsh_parity

pytestmark = pytest.mark.gpu


def _draw(seed, n, d, m, nq, grid):
    rng = np.random.default_rng(seed)
    X = (rng.integers(0, 4, size=(n, d)) if grid else rng.standard_normal((n, d)) * 3)
    X = X.astype(np.float32)
    Q = X[rng.integers(0, n, size=nq)] + rng.standard_normal((nq, d)).astype(np.float32) * 0.1
    Q[: nq // 8] += 40.0  # ranges that start with no data
    A = rng.standard_normal((m, d)).astype(np.float32)
    b = (rng.random(m) * 0.5).astype(np.float32)
    return X, np.ascontiguousarray(Q, np.float32), A, b


@pytest.mark.parametrize("n,m,w,grid", [(1, 1, 0.5, False), (7, 127, 0.5, False),
                                        (9, 3, 50.0, False), (500, 127, 0.05, False),
                                        (TILE, 16, 1.0, True), (TILE + 1, 33, 0.5, False),
                                        (2 * TILE - 1, 64, 3.0, True)])
@pytest.mark.parametrize("path", ["levels", "graph"])
def test_level_forms(orc, qwlib, cuda, n, m, w, grid, path):
    X, Q, A, b = _draw(n + m, n, 5, m, 24, grid)
    _full_parity(orc, qwlib, cuda, X, Q, A, b * w, w=w, k=min(n, 5), v=min(60, n), path=path,
                 l=max(1, m // 2))


@pytest.mark.parametrize("nq,d,m", [(1, 1, 1), (31, 63, 7), (33, 65, 9), (64, 64, 8)])
def test_qalsh_few_rows(orc, qwlib, cuda, nq, d, m):
    X, Q, A, _ = _draw(nq + d, 20_000, d, m, nq, False)
    _qalsh_parity(orc, qwlib, cuda, X, Q, A, w=2.0, k=4, v=50, l=max(1, m // 2))
