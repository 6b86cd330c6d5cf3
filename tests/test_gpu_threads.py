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
