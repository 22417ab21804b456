"""The uv extent pass: the farthest point decides which part of the spectrum is
kept, so a point it missed would be sampled at the edge of a window too small."""
import threading

import numpy as np
import pytest
import torch

import oracle
from paper_1709_06999_gb300 import Context, Request, Server

pytestmark = pytest.mark.gpu
# the visibility gates of the two paths (normwise)
TOL = {torch.float32: 1e-5, torch.float64: 1e-12}


@pytest.mark.parametrize("dt", [torch.float32, torch.float64], ids=["f32", "f64"])
@pytest.mark.parametrize("M", [1, 2, 3, 5, 8, 1023, 4097, 350_003])
def test_farthest_point_anywhere(dt, M):
    """One far point among near ones, at the start, in the middle and in the
    remainder behind the vector groups, in aligned and unaligned arrays."""
    rng = np.random.default_rng(M)
    n, dxy = 128, 1e-8
    img = rng.uniform(0, 1, (n, n))
    ctx = Context(0)
    I = torch.as_tensor(img, dtype=dt, device="cuda")
    h = lambda t: t.double().cpu().numpy()  # noqa: E731
    for at in sorted({0, M // 2, M - 1}):
        for skip in (0, 1):
            u, v = (torch.zeros(M + skip, dtype=dt, device="cuda")[skip:] for _ in range(2))
            near = rng.uniform(-0.02, 0.02, (2, M)) / dxy
            u.copy_(torch.as_tensor(near[0]))
            v.copy_(torch.as_tensor(near[1]))
            u[at], v[at] = 0.31 / dxy, -0.27 / dxy
            got = ctx.sample_image(I, dxy, u, v).double().cpu().numpy()
            sel = np.unique(np.r_[at, rng.integers(0, M, 50)])
            ref = oracle.sample_image(h(I), dxy, h(u)[sel], h(v)[sel])
            err = np.abs(got[sel, 0] + 1j * got[sel, 1] - ref)
            assert np.max(err) <= TOL[dt] * img.sum(), (at, skip)
            # the same point decides for a registered observation
            zero = torch.zeros_like(u)
            w = torch.zeros_like(u)
            w[at] = 1
            chi2 = ctx.chi2_image(I, dxy, ctx.register(u, v, zero, zero, w)).item()
            one = np.abs(ref[list(sel).index(at)]) ** 2
            assert abs(chi2 - one) <= 4 * TOL[dt] * img.sum() * np.sqrt(one) + TOL[dt] ** 2 * img.sum() ** 2


@pytest.mark.parametrize("dt", [torch.float32, torch.float64], ids=["f32", "f64"])
def test_nonfinite_points_and_near_ties(dt):
    rng = np.random.default_rng(7)
    n, dxy, M = 64, 1e-8, 5003
    I = torch.as_tensor(rng.uniform(0, 1, (n, n)), dtype=dt, device="cuda")
    a = rng.uniform(0, 2 * np.pi, M)
    u = torch.as_tensor(0.4 / dxy * np.cos(a), dtype=dt, device="cuda")  # one radius, many roundings
    v = torch.as_tensor(0.4 / dxy * np.sin(a), dtype=dt, device="cuda")
    ctx = Context(0)
    ref = ctx.sample_image(I, dxy, u, v)
    for bad in (float("nan"), float("inf")):
        u2 = u.clone()
        u2[17] = bad
        got = ctx.sample_image(I, dxy, u2, v)
        keep = torch.arange(M, device="cuda") != 17
        assert torch.isnan(got[17]).all()
        # a NaN point is left out of the extent, an infinite one keeps the whole plane
        assert torch.allclose(got[keep], ref[keep], rtol=0, atol=TOL[dt] * I.sum().item())


def test_registrations_from_several_threads():
    """Observations of different reach registered on one server at once: each
    keeps its own extent (a chi-square equal to that of a context of its own)."""
    n, dxy, M = 256, 1e-8, 40_001
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    I = torch.rand((n, n), generator=g, device="cuda")
    data = []
    for k in range(16):
        a = torch.rand((5, M), generator=g, device="cuda")
        r = (0.02 + 0.028 * k) / dxy
        data.append([(a[0] - 0.5) * r, (a[1] - 0.5) * r, a[2], a[3], a[4]])
    torch.cuda.synchronize()
    server = Server(0)
    for _ in range(4):
        obs = [None] * len(data)
        go = threading.Barrier(len(data))

        def work(k):
            go.wait()
            obs[k] = server.add_data(*data[k])

        ts = [threading.Thread(target=work, args=(k,)) for k in range(len(data))]
        for t in ts:
            t.start()
        for t in ts:
            t.join()
        got = [server.wait(server.submit(Request(o, image=I, dxy=dxy)))[0] for o in obs]
        ctx = Context(0)
        want = [ctx.chi2_image(I, dxy, ctx.register(*d)).item() for d in data]
        assert got == want
    server.close()
