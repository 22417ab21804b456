"""Float images of 8192 pixels: registered observations with wide windows take the
row pass two rows to a block, narrow ones one row; the column count decides."""
import numpy as np
import pytest
import torch

import oracle
from paper_1709_06999_gb300 import Context, Request

pytestmark = pytest.mark.gpu
N, DXY = 8192, 1e-9
# farthest point in cells of the grid: windows of 255, 256, 257 and 258 columns
# (cells + 4, the pairs begin at 257), and the whole half plane
REACH = (251.5, 252.5, 253.5, 254.5, 0.49 * N)
FWHM = 0.6 * N * DXY
GEO = dict(dRA=2e-8, dDec=-1e-7, PA=0.4)
M = 1501


@pytest.fixture(scope="module")
def case():
    """Image, points and the FP64 oracle's visibilities without and with a beam."""
    rng = np.random.default_rng(8)
    img = rng.uniform(0, 1, (N, N)).astype(np.float32)
    x = (np.arange(N) - N // 2) / N
    img *= np.exp(-0.5 * (x / 0.1) ** 2).astype(np.float32)[:, None]
    uv = []
    for cells in REACH:
        r = cells * np.sqrt(rng.uniform(0, 1, M))
        a = rng.uniform(0, 2 * np.pi, M)
        r[7] = cells  # the farthest, at 45 degrees
        a[7] = np.pi / 4
        uv.append([(r * f(a) / (N * DXY)).astype(np.float32) for f in (np.cos, np.sin)])
    u, v = (np.concatenate([p[k] for p in uv]).astype(np.float64) for k in (0, 1))
    vis = [oracle.sample_image(img, DXY, u, v, GEO["dRA"], GEO["dDec"], GEO["PA"], f).reshape(-1, M)
           for f in (0.0, FWHM)]
    return torch.as_tensor(img, device="cuda"), uv, vis


def register(ctx, uv, seed):
    rng = np.random.default_rng(seed)
    host = [*uv, *(rng.standard_normal((2, M)).astype(np.float32) * 100),
            rng.uniform(0.5, 2, M).astype(np.float32)]
    dev = [torch.as_tensor(np.ascontiguousarray(h), device="cuda") for h in host]
    return ctx.register(*dev), dev, [h.astype(np.float64) for h in host[2:]]


@pytest.mark.parametrize("fwhm", [0.0, FWHM], ids=["plain", "beam"])
def test_windows_around_the_rule_and_batches_that_mix_them(case, fwhm):
    img, uv, vis = case
    ctx = Context(0)
    reqs, single, keep = [], [], []
    for k, p in enumerate(uv):
        obs, dev, (re, im, w) = register(ctx, p, k)
        got = ctx.chi2_image(img, DXY, obs, pb_fwhm=fwhm, **GEO).item()
        ref = oracle.chi2(vis[1 if fwhm else 0][k], re, im, w)
        assert abs(got - ref) <= 1e-6 * ref, REACH[k]
        reqs.append(Request(obs, image=img, dxy=DXY, pb_fwhm=fwhm, **GEO))
        single.append(got)
        keep.append(dev)
    # the first request decides for a launch: narrow first, wide first, mixed
    for order in ([0, 1, 2, 3, 4], [4, 3, 2, 1, 0], [2, 0], [0, 2], [4, 0, 4, 0], [1], [3]):
        got = ctx.chi2_batch([reqs[i] for i in order]).cpu().tolist()
        assert got == [single[i] for i in order], order
