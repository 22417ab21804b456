"""The default FFT plan is a rule, the same in every process and whatever the
context's tuning is set to."""
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CODE = """
import torch
from paper_1709_06999_gb300 import Context, get_fft_radix
ctx = Context(0)
ctx.set_batch_tuning({tuning})
u = torch.zeros(5, device="cuda")
out = {{}}
for n in (16, 32, 64, 128, 256, 512, 1024):
    before = get_fft_radix(0, torch.float32, n)
    ctx.sample_image(torch.ones((n, n), device="cuda"), 1e-8, u, u)
    out[n] = before, get_fft_radix(0, torch.float32, n)
print(out)
"""


@pytest.mark.parametrize("tuning", [True, False])
def test_default_plan_of_every_side(tuning):
    p = subprocess.run([sys.executable, "-c", CODE.format(tuning=tuning)], capture_output=True,
                       text=True, timeout=300)
    assert p.returncode == 0, p.stderr
    got = eval(p.stdout.strip().splitlines()[-1])
    for n, (before, after) in got.items():
        if 32 <= n <= 512:  # columns at 8; rows at 8 where that takes no more stages
            assert before == (0, 0), n  # not used yet in that process
            assert after == (8 if n in (64, 128) else 16, 8), n
        else:
            assert before == after == (16, 16), n
