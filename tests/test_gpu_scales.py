"""Data far from the origin and of very small or very large coordinates: the locality
order and the start model's features are those of the same data near the origin and
of unit size."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _mixture(cuda, n=60_000, d=32, seed=11):
    """Clustered data on a grid of 1/8 (a multiple of 2^20 added to it is exact)."""
    import torch
    g = torch.Generator(device=cuda).manual_seed(seed)
    centres = torch.rand((60, d), generator=g, device=cuda) * 20 - 10
    lab = torch.randint(0, 60, (n,), generator=g, device=cuda)
    X = torch.round((centres[lab] + torch.randn((n, d), generator=g, device=cuda)) * 8) / 8
    Q = X[torch.randint(0, n, (200,), generator=g, device=cuda)]
    A = torch.randint(-3, 4, (40, d), generator=g, device=cuda).float()
    b = torch.rand((40,), generator=g, device=cuda) * 4
    return X, Q, A, b


def _live_groups(qwlib, X, Q, A, b, w):
    index = qwlib.Index(X.contiguous(), A, b, w=w, v=200, l=26, bitmaps=True)
    ids = index.query(Q.contiguous(), 1, path="bitmap", loads="direct", profile=True)[0]
    live = index.profile()["bitmap_live_groups"]
    index.free()
    return live, ids


@pytest.mark.parametrize("power", [-80, -64, 60, 100])
def test_order_of_scaled_data(qwlib, cuda, power):
    """Scaling by a power of two scales every sum of the tree and rounds nothing, so
    the groups are the same ones."""
    X, Q, A, b = _mixture(cuda)
    want, _ = _live_groups(qwlib, X, Q, A, b, 4.0)
    s = 2.0 ** power
    live, _ = _live_groups(qwlib, X * s, Q * s, A, b * s, 4.0 * s)
    assert live == want


@pytest.mark.parametrize("offset", [2.0 ** 10, 2.0 ** 20])
def test_order_of_shifted_data(qwlib, cuda, offset):
    """An offset that every coordinate can take without rounding moves all bucket ids
    of a projection alike (whole projection vectors, a whole number of bucket
    widths) and leaves every difference as it was."""
    X, Q, A, b = _mixture(cuda)
    assert bool(((X + offset) - offset == X).all())
    want, _ = _live_groups(qwlib, X, Q, A, b, 4.0)
    live, _ = _live_groups(qwlib, X + offset, Q + offset, A, b, 4.0)
    assert live == want


@pytest.mark.parametrize("scale", [1e-30, 1e-23, 1e-21, 1e-19, 1.0, 1e18, 1e20])
def test_features_at_any_scale(qwlib, cuda, scale):
    """The features are the query over the data's RMS coordinate: three roundings
    (the factor, its narrowing and the product) and an RMS good to 2^-33."""
    import torch
    rng = np.random.default_rng(6)
    X = (rng.standard_normal((3000, 17)) * scale).astype(np.float32)
    X[::3] *= np.float32(2.0 ** -20)
    index = qwlib.Index(*(torch.from_numpy(x).to(cuda) for x in
                          (X, rng.standard_normal((5, 17)).astype(np.float32),
                           np.zeros(5, np.float32))), w=scale, v=10, l=2)
    F = index.features(torch.from_numpy(X[1:9]).to(cuda))[:, :17].cpu().numpy().astype(np.float64)
    rms = np.sqrt(np.mean(X.astype(np.float64) ** 2))
    want = X[1:9].astype(np.float64) / rms
    assert np.all(np.abs(F - want) <= 3 * 2.0 ** -24 * np.abs(want))
    index.free()
