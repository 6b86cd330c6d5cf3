"""Data of very small or very large coordinates: the start model's features are those
of the same data of unit size."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


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
