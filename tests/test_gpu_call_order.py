"""Calls in a row overlap their launches: each must still see everything enqueued
before it, and nothing after it."""
import pytest
import torch

from paper_1709_06999_gb300 import Context

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dt", [torch.float32, torch.float64], ids=["f32", "f64"])
@pytest.mark.parametrize("n,M", [(128, 3001), (1024, 40_000), (2048, 300_001), (4096, 50_000)])
def test_inputs_rewritten_between_calls(dt, n, M):
    """Image, data and points are rewritten in place between calls that nothing
    waits between; every result equals that of the call made alone."""
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    dxy = 1e-8
    img = torch.rand((n, n), generator=g, device="cuda", dtype=dt)
    a = torch.rand((5, M), generator=g, device="cuda", dtype=dt)
    u, v = (a[0] - 0.5) * (0.4 / dxy), (a[1] - 0.5) * (0.4 / dxy)
    re, im, w = a[2].contiguous(), a[3].contiguous(), a[4].contiguous()
    ctx = Context(0)
    obs = ctx.register(u, v, re, im, w)

    def step(k, wait):
        out = []
        if wait:
            torch.cuda.synchronize()
        out.append(ctx.chi2_image(img, dxy, obs, 1e-8, -2e-8, 0.1 * k))
        img.mul_(1.25)
        re.add_(0.5)
        w.mul_(0.75)
        if wait:
            torch.cuda.synchronize()
        out.append(ctx.chi2_image(img, dxy, obs))
        if wait:
            torch.cuda.synchronize()
        out.append(ctx.sample_image(img, dxy, u * (0.5 + 0.1 * k), v))
        img.mul_(0.5)
        return out

    results = []
    for wait in (True, False):
        keep = [t.clone() for t in (img, re, w)]
        got = []
        for k in range(6):
            got += step(k, wait)
        torch.cuda.synchronize()
        results.append([t.clone() for t in got])
        for t, s in zip((img, re, w), keep):
            t.copy_(s)
    for x, y in zip(*results):
        assert torch.equal(x, y)
