"""The double path's integer arithmetic (csrc/gal_fx.cuh) at the places where it
can go wrong: every transform plan, pruned and complete windows, block exponents
at the ends of the double range, zeros, non-finite values, and points on nodes,
on the edges of the grid and beyond it."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_1709_06999_gb300 import Context

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -53


def points(n, dxy, reach, M=2001, seed=0):
    """Random points within reach of the Nyquist frequency, some on nodes and axes."""
    rng = np.random.default_rng(seed)
    du = 1.0 / (n * dxy)
    rho = reach * 0.5 / dxy
    a, r = rng.uniform(0, 2 * math.pi, M), rho * np.sqrt(rng.uniform(0, 1, M))
    u, v = r * np.cos(a), r * np.sin(a)
    k = min(40, M // 4)
    lim = max(1, int(reach * n / 2 * 0.7))
    u[:k], v[:k] = rng.integers(-lim, lim + 1, k) * du, rng.integers(-lim, lim + 1, k) * du
    u[k], v[k], u[k + 1], v[k + 2] = 0.0, 0.0, -0.0, 0.0
    return u, v


def sample(ctx, img, dxy, u, v, *geo):
    d = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")  # noqa: E731
    out = ctx.sample_image(d(img), dxy, d(u), d(v), *geo).cpu().numpy()
    return out[:, 0] + 1j * out[:, 1]


# a position takes three roundings of a value below n cells, and one cell moves a
# visibility by at most 2 max|V|; transform, phase and interpolation add a few
# dozen roundings relative to the largest value
def tol(n):
    return (6 * n + 64) * EPS


@pytest.mark.parametrize("n", [16, 32, 64, 128, 256, 512, 1024, 2048, 4096])
@pytest.mark.parametrize("reach", [0.02, 0.3, 0.95])
def test_every_plan_against_the_oracle(n, reach):
    rng = np.random.default_rng(n)
    img = rng.uniform(0, 1, (n, n)) * np.exp(-8 * np.linspace(-1, 1, n) ** 2)[:, None]
    dxy = 1e-8
    u, v = points(n, dxy, reach)
    geo = (3.3e-8 * n / 16, -2.1e-8 * n / 16, 0.7)
    got = sample(Context(0), img, dxy, u, v, *geo)
    ref = oracle.sample_image(img, dxy, u, v, *geo)
    assert np.max(np.abs(got - ref)) <= tol(n) * np.max(np.abs(ref))


@pytest.mark.parametrize("k", [-960, -400, 400, 900])
def test_scaling_by_a_power_of_two_is_exact(k):
    rng = np.random.default_rng(1)
    img = rng.standard_normal((128, 128)) * 10.0 ** rng.uniform(-6, 0, (128, 128))
    u, v = points(128, 1e-8, 0.9)
    ctx = Context(0)
    a = sample(ctx, img, 1e-8, u, v, 1e-8, 2e-8, 0.3)
    b = sample(ctx, img * 2.0 ** k, 1e-8, u, v, 1e-8, 2e-8, 0.3)
    assert np.array_equal(b.real, a.real * 2.0 ** k) and np.array_equal(b.imag, a.imag * 2.0 ** k)


@pytest.mark.parametrize("n", [64, 2048])
def test_rows_of_very_different_size(n):
    """One row 1e150 times the others (its block exponent is its own), a row of
    zeros, a single pixel, and pixels that vanish beside their row's largest."""
    rng = np.random.default_rng(2)
    img = rng.uniform(0, 1, (n, n))
    img[n // 3] *= 1e150
    img[n // 4] = 0.0
    img[n // 5] = 0.0
    img[n // 5, n // 7] = 1e150
    img[n // 6, ::2] *= 1e-310
    u, v = points(n, 1e-8, 0.2)
    got = sample(Context(0), img, 1e-8, u, v)
    ref = oracle.sample_image(img, 1e-8, u, v)
    assert np.max(np.abs(got - ref)) <= tol(n) * np.max(np.abs(ref))


def test_zero_and_nonfinite():
    ctx = Context(0)
    n, dxy = 64, 1e-8
    u, v = points(n, dxy, 0.9, M=101)
    assert np.all(sample(ctx, np.zeros((n, n)), dxy, u, v) == 0)
    for bad in (np.nan, np.inf):
        img = np.ones((n, n))
        img[5, 9] = bad
        assert np.all(~np.isfinite(sample(ctx, img, dxy, u, v)))
    img = np.random.default_rng(3).uniform(0, 1, (n, n))
    ref = oracle.sample_image(img, dxy, u, v, 1e-8, 1e-8, 0.2)
    uu, vv = u.copy(), v.copy()
    uu[3], vv[7], uu[11] = np.nan, np.inf, -np.inf
    got = sample(ctx, img, dxy, uu, vv, 1e-8, 1e-8, 0.2)
    hit = np.isin(np.arange(len(u)), (3, 7, 11))
    assert np.all(np.isnan(got[hit].real)) and np.all(np.isnan(got[hit].imag))
    # a NaN extent keeps the whole plane: the other points are the oracle's still
    assert np.max(np.abs(got[~hit] - ref[~hit])) <= tol(n) * np.max(np.abs(ref))


@pytest.mark.parametrize("n", [32, 512])
def test_beyond_the_grid(n):
    """Points on and beyond the edges of the node range take the edge value."""
    rng = np.random.default_rng(4)
    img, dxy = rng.uniform(0, 1, (n, n)), 1e-8
    du = 1.0 / (n * dxy)
    e = np.array([n / 2 - 1, n / 2 - 0.5, n / 2, n / 2 + 0.5, n, 3.7 * n, 5000.25, 1e6, 1e12]) * du
    u, v = (a.ravel() for a in np.meshgrid(np.concatenate([e, -e]), np.concatenate([e, -e])))
    got, ref = sample(Context(0), img, dxy, u, v), oracle.sample_image(img, dxy, u, v)
    assert np.max(np.abs(got - ref)) <= tol(n) * np.sum(img)
