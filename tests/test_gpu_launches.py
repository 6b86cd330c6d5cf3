"""The launch counts of qw_index_profile are the kernels launched: against the CUDA
profiler's record of a call, and in graph mode against the host-driven loop's count
per level."""
import pytest

import workloads

pytestmark = pytest.mark.gpu


def _index(qwlib, cuda, **kw):
    import torch
    wl = workloads.make_workload("mix10k_d32", seed=31, n=40_000, nq=400, n_clusters=30)
    X, A, b = (torch.from_numpy(a).to(cuda) for a in (wl.X, wl.A, wl.b))
    return qwlib.Index(X, A, b, w=4.0, v=60, **kw), torch.from_numpy(wl.Q).to(cuda)


def _counted(index, Q, **kw):
    import torch
    from torch.profiler import ProfilerActivity, profile
    index.query(Q, 5, **kw)
    torch.cuda.synchronize()
    for _ in range(2):  # (a process's first session may start late)
        index.profile(reset=True)
        with profile(activities=[ProfilerActivity.CUDA]) as prof:
            index.query(Q, 5, **kw)
            torch.cuda.synchronize()
    seen = [e.name for e in prof.events()
            if e.device_type == torch.autograd.DeviceType.CUDA and "qw::" in e.name]
    return index.profile(reset=True)["launches"], seen


@pytest.mark.parametrize("nq", [16, 300])
@pytest.mark.parametrize("kw", [dict(path="levels"), dict(path="levels", order="signature"),
                                dict(path="bitmap", loads="direct"),
                                dict(path="bitmap", loads="fused", batch=70),
                                dict(path="bitmap", loads="tma", rerank="bf16"),
                                dict(path="cluster")], ids=repr)
def test_launches_of_a_call(qwlib, cuda, nq, kw):
    index, Q = _index(qwlib, cuda, bitmaps=True, shadow_bf16=True)
    launches, seen = _counted(index, Q[:nq].contiguous(), **kw)
    assert seen and sum(launches.values()) == len(seen)
    index.free()


@pytest.mark.parametrize("nq", [16, 300])
@pytest.mark.parametrize("kw", [dict(path="levels"), dict(path="bitmap", loads="direct"),
                                dict(path="bitmap", loads="fused"),
                                dict(path="bitmap", loads="tma")], ids=repr)
def test_launches_in_graph_mode(qwlib, cuda, nq, kw):
    """One batch: the loop's three first kernels, then per level its counting
    kernels, the decision and the loop's step."""
    index, Q = _index(qwlib, cuda, bitmaps=True)
    Q = Q[:nq].contiguous()
    host, _ = _counted(index, Q, **kw)
    per_level, rest = divmod(host["level"] + host["bucket"], host["decide"])
    assert rest == 0
    graph, _ = _counted(index, Q, graph=True, **kw)
    levels, rest = divmod(graph["decide"] - 3, 2)
    assert rest == 0 and 0 < levels <= host["decide"]
    assert graph["level"] == levels * per_level and graph["bucket"] == 0
    index.free()
