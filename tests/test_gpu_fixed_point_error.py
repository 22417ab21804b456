"""How far the double path's transforms are from the exact spectrum, root mean
square, at nodes near the origin: dense sequences (noise), where every pixel is as
large as every other, are the hard ones for a common power of two."""
import math

import numpy as np
import pytest
import torch

from paper_1709_06999_gb300 import Context

pytestmark = pytest.mark.gpu
K = 24  # half width of the window of nodes, in cells


def image(kind, n, rng):
    """Integers below 2^20, so that their products with 21-bit digits add up exactly."""
    if kind == "noise":
        return np.rint(np.clip(rng.standard_normal((n, n)), -7, 7) * 2.0 ** 17)
    if kind == "positive":
        return np.floor(rng.uniform(0, 1, (n, n)) * 2.0 ** 19)
    x = (np.arange(n) - n // 2) / n
    r = np.hypot(x[None, :] - 0.03, (x[:, None] + 0.01) * 1.7)
    return np.rint(2.0 ** 19 * (np.exp(-0.5 * (r / 0.02) ** 2) + 0.5 * np.exp(-r / 0.03)))


def exact_nodes(img):
    """G[l, k] = sum_ij x_ij exp(-2 pi i (l i + k j) / n), |l| <= K, 0 <= k <= K: the
    sums over j exactly (63-bit factors in three digits), those over i in extended
    precision."""
    n = img.shape[0]
    x = np.fft.fftshift(img)
    m = np.arange(n)
    turn = 2 * np.longdouble("3.14159265358979323846264338327950288") / n
    c, s = np.cos(turn * m), -np.sin(turn * m)
    jk = np.outer(m, np.arange(K + 1)) % n
    A = []
    for w in (c[jk], s[jk]):
        acc = np.zeros((n, K + 1), dtype=np.longdouble)
        for bits in (21, 42, 63):
            d = np.rint(np.ldexp(w, bits)).astype(np.float64)  # below 2^21
            w = w - np.ldexp(d.astype(np.longdouble), -bits)
            acc += np.ldexp((x @ d).astype(np.longdouble), -bits)
        A.append(acc)
    il = np.outer(np.arange(-K, K + 1), m) % n
    C, S = c[il], s[il]
    return (C @ A[0] - S @ A[1]), (C @ A[1] + S @ A[0])


@pytest.mark.parametrize("kind,n", [(k, n) for n in (64, 512, 1024, 2048, 4096)
                                    for k in ("noise", "positive", "smooth")] + [("noise", 8192)])
def test_error_is_that_of_double_arithmetic(kind, n):
    """An FP64 transform of n x n points rounds each of the 2 log2(n) levels of its
    sums at 2^-53 of their size: 2^-53 sqrt(2 log2 n) over the rms visibility."""
    img = image(kind, n, np.random.default_rng(n))
    dxy = 2.0 ** -27  # a power of two: the nodes' positions are exact
    k, l = np.meshgrid(np.arange(K + 1), np.arange(-K, K + 1))
    u, v = (torch.as_tensor(a.ravel() / (n * dxy), device="cuda") for a in (k, l))
    got = Context(0).sample_image(torch.as_tensor(img, device="cuda"), dxy, u, v).cpu().numpy()
    re, im = exact_nodes(img)
    dr, di = got[:, 0] - re.ravel(), got[:, 1] - im.ravel()
    err = math.sqrt(float(np.sum(dr * dr + di * di) / np.sum(re * re + im * im)))
    assert err <= 2.0 ** -53 * math.sqrt(2 * math.log2(n)), err


@pytest.mark.parametrize("n", [64, 128, 256, 512, 1024, 2048, 4096, 8192])
def test_sums_as_large_as_they_can_be(n):
    """Images whose values add up without cancelling, in every stage: the bound that
    the integers are scaled to is reached, and none of them may wrap."""
    ctx = Context(0)
    dxy = 2.0 ** -27
    k, l = np.meshgrid(np.arange(K + 1), np.arange(-K, K + 1))
    u, v = (torch.as_tensor(a.ravel() / (n * dxy), device="cuda") for a in (k, l))
    i = np.arange(n)
    ones = np.ones((n, n))
    wave = np.cos(2 * np.pi * ((3 * i[:, None] + 5 * i[None, :]) % n) / n)
    corner = np.zeros((n, n))
    corner[0] = corner[:, n // 4] = 1.0  # a full row and a full column
    spike = np.rint(wave * 3)
    spike[n // 3, n // 5] = 2.0 ** 20 - 1
    for img in (ones * (2 ** 20 - 1), ones * 2 ** 19, np.rint(wave * (2 ** 20 - 1)),
                np.where((i[:, None] + i[None, :]) % 2, -1.0, 1.0) * (2 ** 20 - 1),
                corner * (2 ** 20 - 1), spike):
        got = ctx.sample_image(torch.as_tensor(img, device="cuda"), dxy, u, v).cpu().numpy()
        re, im = exact_nodes(img)
        err = np.max(np.hypot(got[:, 0] - re.ravel(), got[:, 1] - im.ravel()).astype(np.float64))
        # every level rounds at 2^-53 of the largest value the level can have
        assert err <= 2 * math.log2(n) * 2.0 ** -53 * np.abs(img).sum()
