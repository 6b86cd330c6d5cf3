"""The autotuner tries a setting only where something reads it: the tiles per warp are
the fused bitmap kernel's alone."""
import pytest

import workloads

pytestmark = pytest.mark.gpu


def test_tile_shapes_only_with_fused_loads(qwlib, cuda):
    import torch
    wl = workloads.make_workload("mix10k_d32", seed=26, n=20_000, nq=40, n_clusters=20)
    X, A, b, Q = (torch.from_numpy(a).to(cuda) for a in (wl.X, wl.A, wl.b, wl.Q))
    index = qwlib.Index(X, A, b, w=4.0, v=40, bitmaps=True)
    best, trials = index.autotune(Q, 5, reps=1)
    for t in [best] + [t for t, _ in trials]:
        assert t["tiles_per_warp"] == 0 or t["loads"] == "fused"
    assert any(t["loads"] == "direct" for t, _ in trials)
    index.free()
