"""Registrations on one context from several threads and streams do not wait for
one another."""
import threading
import time

import pytest
import torch

from paper_1709_06999_gb300 import Context

pytestmark = pytest.mark.gpu


def test_a_busy_stream_holds_up_its_own_registration_only():
    """Four registrations wait on streams that are busy for some time; one on an idle
    stream is done long before, and all of them keep their own extent."""
    dxy, n, M, busy = 1e-8, 64, 5003, 4
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    I = torch.rand((n, n), generator=g, device="cuda")
    data = []
    for k in range(busy + 1):
        a = torch.rand((5, M), generator=g, device="cuda")
        r = (0.1 + 0.08 * k) / dxy
        data.append([(a[0] - 0.5) * r, (a[1] - 0.5) * r, a[2], a[3], a[4]])
    ctx = Context(0)
    first = ctx.register(*data[0])  # loads the kernels (kept: dropping it waits for the device)
    streams = [torch.cuda.Stream() for _ in data]
    torch.cuda.synchronize()
    obs, done = [None] * len(data), [0.0] * len(data)
    started = threading.Barrier(busy + 1)

    def work(k):
        with torch.cuda.stream(streams[k]):
            if k < busy:
                torch.cuda._sleep(600_000_000)  # about 0.3 s
            started.wait()
            if k == busy:
                time.sleep(0.05)  # the others are waiting for their streams by now
            obs[k] = ctx.register(*data[k])
            done[k] = time.perf_counter()

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(data))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert done[busy] < min(done[:busy]) - 0.05
    first.close()
    alone = Context(0)
    for o, d in zip(obs, data):
        want = alone.chi2_image(I, dxy, alone.register(*d)).item()
        assert ctx.chi2_image(I, dxy, o).item() == want
