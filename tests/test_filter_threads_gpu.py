"""Filters of different radii from two host threads, each on a stream of its own: the shared-memory limit that a launch
needs is state of the kernel on the device, so one thread's call must not lower it under another's.  Each call's
result is the one that the same call gives alone, bit for bit (the kernels add in a fixed order)."""
import threading

import pytest

from test_filter_gpu import N  # noqa: F401

pytestmark = pytest.mark.gpu


def test_radii_of_concurrent_threads(N):  # noqa: F811
    import torch
    shape, calls = (9, 11, 13), 3000
    x = torch.rand(shape, device="cuda")

    def filtered(R, stream):
        rt, rb, g = (torch.empty_like(x) for _ in range(3))
        N.fdtd_filter_project(x, rt, rb, R, 6.0, 0.5, stream.cuda_stream)
        N.fdtd_filter_project_grad(rt, x, g, R, 6.0, 0.5, stream.cuda_stream)
        return rt, rb, g

    radii = (2.0, 12.0, 12.0)
    streams = [torch.cuda.Stream() for _ in radii]
    torch.cuda.synchronize()
    want, got, errors = [], [None] * len(radii), []
    for R, s in zip(radii, streams):
        with torch.cuda.stream(s):
            want.append(filtered(R, s))
        s.synchronize()

    def work(i):
        try:
            with torch.cuda.stream(streams[i]):
                for _ in range(calls):
                    got[i] = filtered(radii[i], streams[i])
            streams[i].synchronize()
        except N.FdtdError as e:
            errors.append((radii[i], str(e)))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(radii))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors
    for a, b in zip(got, want):
        assert all(torch.equal(p, q) for p, q in zip(a, b))
