"""Chi-square over few points in double: the points are spread over the GPU's SMs,
in single calls and in batches alike, from arrays of any alignment."""
import numpy as np
import pytest
import torch

import oracle
from paper_1709_06999_gb300 import Context, Request

pytestmark = pytest.mark.gpu
DXY = 1e-8


def observation(ctx, n, M, reach, skip, seed):
    """Registered arrays (behind `skip` further values: 1 misaligns them) and their host copies."""
    rng = np.random.default_rng(seed)
    a = rng.uniform(0, 2 * np.pi, M)
    r = reach / DXY * np.sqrt(rng.uniform(0, 1, M))
    host = [r * np.cos(a), r * np.sin(a), rng.standard_normal(M), rng.standard_normal(M),
            rng.uniform(0.5, 2, M)]
    dev = []
    for x in host:
        t = torch.zeros(M + skip, dtype=torch.float64, device="cuda")[skip:]
        t.copy_(torch.as_tensor(x))
        dev.append(t)
    return ctx.register(*dev), dev, host


# 128 groups of two points to a block, and the largest counts that are spread:
# 152 blocks with the window in shared memory (side 64), 608 through L2 (side 256)
@pytest.mark.parametrize("n,reach", [(64, 0.4), (256, 0.45)])
def test_counts_around_block_edges(n, reach):
    rng = np.random.default_rng(n)
    img = rng.uniform(0, 1, (n, n))
    I = torch.as_tensor(img, device="cuda")
    ctx = Context(0)
    reqs, single = [], []
    for M in (1, 2, 3, 63, 255, 256, 257, 3001, 38_911, 38_913, 155_648, 155_651, 311_297):
        for skip in (0, 1):
            obs, keep, host = observation(ctx, n, M, reach, skip, M + skip)
            geo = dict(dRA=1e-8, dDec=-3e-8, PA=0.3)
            got = ctx.chi2_image(I, DXY, obs, **geo).item()
            ref = oracle.chi2_image(img, DXY, *host, 1e-8, -3e-8, 0.3)
            assert abs(got - ref) <= 1e-12 * ref, (M, skip)
            reqs.append(Request(obs, image=I, dxy=DXY, **geo))
            single.append(got)
    assert ctx.chi2_batch(reqs).cpu().tolist() == single
    for part in (reqs[:1], reqs[6:9], reqs[::-1]):  # other launches, other numbers of blocks
        want = [single[reqs.index(r)] for r in part]
        assert ctx.chi2_batch(part).cpu().tolist() == want


@pytest.mark.parametrize("skip", [0, 1], ids=["aligned", "misaligned"])
def test_few_points_take_less_time_than_many(skip):
    """The FP64 work of 2e4 points on a GPU's SMs is a tenth of that of 2e5.  Packed
    into full blocks of 1024 threads, one to an SM, both would take the same time
    (33.2 and 34.9 us a call); spread they take 22.6 and 33.0 us."""
    ctx = Context(0)
    n = 64
    I = torch.rand((n, n), dtype=torch.float64, device="cuda")

    def us(M):
        obs, keep, _ = observation(ctx, n, M, 0.4, skip, M)
        best = []
        for _ in range(7):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            for _ in range(20):
                ctx.chi2_image(I, DXY, obs)
            a.record()
            for _ in range(200):
                ctx.chi2_image(I, DXY, obs)
            b.record()
            torch.cuda.synchronize()
            best.append(a.elapsed_time(b) / 200 * 1e3)
        return min(best)

    few, many = us(20_001 - skip), us(300_001 - skip)
    assert few <= 0.85 * many, (few, many)
