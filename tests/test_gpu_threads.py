"""Calls from several threads at once (the binding releases the interpreter lock),
each on its own index and stream, whose kernels ask for different amounts of
shared memory: every call succeeds and answers as it does alone."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _together(jobs):
    """Run the jobs on a thread each; the first exception is raised here."""
    errors = []

    def body(job):
        try:
            job()
        except Exception as e:  # noqa: BLE001 - handed to the test's thread
            errors.append(e)

    threads = [threading.Thread(target=body, args=(job,)) for job in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    if errors:
        raise errors[0]


def test_index_builds(qwlib, cuda):
    """Builds of indexes whose bucket spans, and so the sort's counting tables,
    differ."""
    import torch
    g = torch.Generator(device=cuda).manual_seed(3)
    A = torch.randn((8, 8), generator=g, device=cuda)
    b = torch.rand((8,), generator=g, device=cuda) * 4
    data = [torch.randn((3000, 8), generator=g, device=cuda) * s for s in (1.0, 20.0, 60.0, 90.0)]

    def build(X):
        index = qwlib.Index(X, A, b, w=4.0, v=30, l=2)
        out = index.export()
        index.free()
        return out

    want = [build(X) for X in data]
    assert len({int(w[1].max()) for w in want}) == 4 and max(int(w[1].max()) for w in want) < 1023
    torch.cuda.synchronize()

    def job(X, ref):
        def run():
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(200):
                    for x, y in zip(build(X), ref):
                        assert np.array_equal(x, y)
        return run

    _together([job(X, ref) for X, ref in zip(data, want)])


@pytest.mark.parametrize("kw", [dict(path="levels"), dict(path="cluster"),
                                dict(path="bitmap", loads="direct"),
                                dict(path="bitmap", loads="direct", rerank="bf16"),
                                dict(path="levels", rerank="bf16_tc")],
                         ids=["levels", "cluster", "bitmap", "bf16", "bf16_tc"])
def test_queries(qwlib, cuda, kw):
    """Workloads with different k + v (candidate slots per block), numbers of
    projections and of id tiles."""
    import torch
    g = torch.Generator(device=cuda).manual_seed(4)
    jobs = []
    for n, m, k, v in ((5000, 10, 5, 20), (9000, 12, 10, 1500), (70_000, 16, 10, 4000),
                       (40_000, 40, 1, 300)):
        X = torch.randn((n, 16), generator=g, device=cuda)
        Q = (X[:40] + 0.1).contiguous()
        A = torch.randn((m, 16), generator=g, device=cuda)
        b = torch.rand((m,), generator=g, device=cuda)
        index = qwlib.Index(X, A, b, w=1.0, v=v, l=m // 2, bitmaps=True, shadow_bf16=True)
        ref = index.query(Q, k, stats=True, **kw)

        def run(index=index, Q=Q, k=k, ref=ref):
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(100):
                    for x, y in zip(index.query(Q, k, stats=True, **kw), ref):
                        assert torch.equal(x, y)

        jobs.append((index, run))
    torch.cuda.synchronize()
    _together([run for _, run in jobs])
    for index, _ in jobs:
        index.free()


def test_hash_and_start_model(orc, qwlib, cuda):
    """Tensor-core projections of few and of many columns, start models of
    different sizes."""
    import torch
    g = torch.Generator(device=cuda).manual_seed(5)
    jobs = []
    for m in (16, 127, 33, 96):
        X = torch.randn((300, 24), generator=g, device=cuda)
        A = torch.randn((m, 24), generator=g, device=cuda)
        b = torch.rand((m,), generator=g, device=cuda)
        want = torch.from_numpy(orc.hash(*(t.cpu().numpy() for t in (X, A, b)), 1.0)).to(cuda)

        def run(X=X, A=A, b=b, want=want):
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(200):
                    assert torch.equal(qwlib.hash(X, A, b, 1.0, tensor_cores=True)[0], want)

        jobs.append(run)
    models = []
    for n_in, hidden, tc in ((64, 256, True), (576, 256, True)):
        model = qwlib.Mlp(n_in, hidden, 16)
        model.set_params(qwlib.mlp_init(n_in, hidden, 16, seed=n_in))
        F = torch.randn((200, n_in), generator=g, device=cuda)
        ref = model.predict(F, tensor_cores=tc)
        models.append(model)

        def run2(model=model, F=F, ref=ref, tc=tc):
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(200):
                    assert torch.equal(model.predict(F, tensor_cores=tc), ref)

        jobs.append(run2)
    torch.cuda.synchronize()
    _together(jobs)
    for model in models:
        model.free()
