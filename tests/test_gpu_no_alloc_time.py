"""The allocation-free chi-square rebuilds its twiddle tables in every call: that
must not become a large part of the call."""
import ctypes as ct

import pytest
import torch

from paper_1709_06999_gb300 import _native

pytestmark = pytest.mark.gpu


def test_tables_cost_little():
    """Sides 16 and 256 differ by the passes' work and by the tables': 25.6 and 31.3
    us a call with the tables side by side, 27.1 and 41.5 with one after the other.
    Twenty calls in a graph, so that the host does not count."""
    lib = _native.load()
    M, dxy = 4096, 1e-8
    d = [torch.rand(M, device="cuda") for _ in range(5)]
    for t in d[:2]:
        t.sub_(0.5).mul_(0.6 / dxy)
    out = torch.empty((), dtype=torch.float64, device="cuda")

    def us(n):
        img = torch.rand((n, n), device="cuda")

        def call():
            stream = ct.c_void_p(torch.cuda.current_stream().cuda_stream)
            st = lib.gal_chi2_image_noalloc_f32(
                img.data_ptr(), n, dxy, 0.0, 0.0, 0.0, *[t.data_ptr() for t in d], M,
                out.data_ptr(), stream)
            assert st == 0

        call()
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            for _ in range(20):
                call()
        times = []
        for _ in range(7):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            graph.replay()
            a.record()
            for _ in range(5):
                graph.replay()
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b) / 100 * 1e3)
        return min(times)

    small, large = us(16), us(256)
    assert large <= 1.33 * small, (small, large)
