"""Calls that follow one another with nothing between them: a float image's row pass
is launched while the previous call's gather still runs and shares its workspace
with it.  Every result equals that of the same call made alone."""
import pytest
import torch

from paper_1709_06999_gb300 import Context, Request
import paper_1709_06999_gb300 as gal

pytestmark = pytest.mark.gpu
DXY = 1e-8


def observation(ctx, g, n, M, reach, dt):
    a = torch.rand((5, M), generator=g, device="cuda", dtype=dt)
    r = 2 * reach / DXY
    arrays = [((a[0] - 0.5) * r).contiguous(), ((a[1] - 0.5) * r).contiguous(), a[2].contiguous(),
              a[3].contiguous(), (a[4] + 0.5).contiguous()]
    return ctx.register(*arrays), arrays


def calls(ctx, sides, dt):
    """Closures of every entry point over images of the given sides: different
    images, geometries, observations, narrow windows and wide ones."""
    g = torch.Generator(device="cuda")
    g.manual_seed(len(sides))
    out = []
    for k, n in enumerate(sides):
        img = [torch.rand((n, n), generator=g, device="cuda", dtype=dt) for _ in range(2)]
        prof = torch.rand(500, generator=g, device="cuda", dtype=dt)
        near, na = observation(ctx, g, n, 200_003 + 1000 * k, 0.01, dt)
        far, fa = observation(ctx, g, n, 30_001 + 1000 * k, 0.3, dt)
        geo = dict(dRA=(k + 1) * 1e-8, dDec=-2e-8, PA=0.2 * k)
        src = ([1e-8, -3e-8, 5e-8], [0.0, 2e-8, -1e-8], [1.0, 0.5, 0.25])
        dR = 0.4 * n * DXY / 500
        out += [
            lambda i=img, o=far, q=geo: ctx.chi2_image(i[0], DXY, o, **q),
            lambda i=img, o=near: ctx.chi2_image(i[1], DXY, o),
            lambda i=img, o=far, s=src: ctx.chi2_image_multi(i[0], DXY, o, *s),
            lambda i=img, o=near, q=geo: ctx.chi2_image(i[0], DXY, o, **q),
            lambda i=img, a=fa: ctx.sample_image(i[1], DXY, a[0], a[1]),
            lambda i=img, o=near, q=geo: ctx.chi2_image(i[1], DXY, o, **q),
            lambda i=img, o=far, f=0.5 * n * DXY: ctx.chi2_image(i[0], DXY, o, pb_fwhm=f),
            lambda i=img, o=far: ctx.chi2_image(i[1], DXY, o),
            lambda p=prof, o=far, n=n, d=dR: ctx.chi2_profile(p, d / 2, d, n, DXY, o, inc=0.3),
            lambda i=img, o=near: ctx.chi2_image(i[0], DXY, o),
            lambda p=prof, a=na, n=n, d=dR: ctx.sample_profile(p, d / 2, d, n, DXY, a[0], a[1]),
            lambda i=img, o=far: ctx.chi2_image(i[0], DXY, o),
            lambda i=img, o=(near, far): ctx.chi2_batch([Request(x, image=i[0], dxy=DXY) for x in o]),
            lambda i=img, o=near: ctx.chi2_image(i[1], DXY, o),
        ]
        if n <= 4096:
            out += [lambda i=img, o=far: ctx.chi2_image(i[0], DXY, o, full_plane=True),
                    lambda i=img, o=near: ctx.chi2_image(i[1], DXY, o),
                    lambda i=img, a=fa: gal.chi2_image(i[0], DXY, *a),
                    lambda i=img, o=far: ctx.chi2_image(i[1], DXY, o)]
    return out


def alone(fns):
    res = []
    for f in fns:
        torch.cuda.synchronize()
        res.append(f().clone())
    torch.cuda.synchronize()
    return res


@pytest.mark.parametrize("dt,sides", [
    (torch.float32, (2048, 4096, 2048)), (torch.float32, (8192, 1024)),
    (torch.float32, (256, 512, 128, 4096)), (torch.float64, (256, 2048, 1024))],
    ids=["f32-2048-4096", "f32-8192", "f32-small", "f64"])
def test_calls_in_a_row(dt, sides):
    ctx = Context(0)
    fns = calls(ctx, sides, dt)
    want = alone(fns)
    order = list(range(len(fns)))
    for step in (1, 5, 11):  # neighbours of the same side, then sides alternating
        seq = [order[(i * step) % len(order)] for i in range(len(order))]
        torch.cuda.synchronize()
        got = [fns[i]() for i in seq]
        torch.cuda.synchronize()
        for i, x in zip(seq, got):
            assert torch.equal(x, want[i]), i
    ctx.check()


def test_same_calls_over_and_over():
    """The listed pair of the large image: no call in between, no allocation."""
    ctx = Context(0)
    fns = calls(ctx, (4096,), torch.float32)
    want = alone(fns[:4])
    got = [[f() for f in fns[:4]] for _ in range(25)]
    torch.cuda.synchronize()
    for row in got:
        for x, y in zip(row, want):
            assert torch.equal(x, y)


def test_two_streams_with_a_context_each():
    """Contexts do not share workspace: calls on two streams may overlap."""
    ctxs = [Context(0), Context(0)]
    fns = [calls(c, (2048, 512), torch.float32) for c in ctxs]
    want = [alone(f) for f in fns]
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    torch.cuda.synchronize()
    got = [[], []]
    for i in range(len(fns[0])):
        for s in (0, 1):
            with torch.cuda.stream(streams[s]):
                j = (i * (1 + 4 * s)) % len(fns[s])
                got[s].append((j, fns[s][j]()))
    torch.cuda.synchronize()
    for s in (0, 1):
        for j, x in got[s]:
            assert torch.equal(x, want[s][j]), (s, j)
