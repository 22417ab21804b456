"""Shared memory that a bulk copy refills has been used by ordinary loads and
stores before.  A block barrier does not order those against the copy (another
proxy); a proxy fence does.  What a missing fence does to a result depends on the
hardware's timing, so the sources are checked, not results."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1709_06999_gb300", "csrc")


def refills():
    """(file, line, the lines since the loop's last wait) of every refill of a ring."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cuh"))):
        lines = open(path).read().splitlines()
        for i, line in enumerate(lines):
            if not re.search(r"\bissue\((it|grp) \+", line):
                continue
            start = max(k for k in range(i) if "mbar_wait(" in lines[k])
            yield os.path.basename(path), i + 1, lines[start:i]


def test_there_are_rings():
    assert {f for f, _, _ in refills()} == {"gal_fx_kernels.cuh", "gal_kernels.cuh", "gal_plane.cuh"}


@pytest.mark.parametrize("where", list(refills()), ids=lambda w: f"{w[0]}:{w[1]}")
def test_refill_is_fenced(where):
    """A proxy fence stands between the slot's last use and its refill: before the
    barrier (by every thread: it covers their stores) or, where the slot was only
    read, after it."""
    _, _, body = where
    code = [re.sub(r"//.*", "", s) for s in body]
    fence = [k for k, s in enumerate(code) if "fence_proxy_async_smem()" in s]
    sync = [k for k, s in enumerate(code) if re.search(r"__syncthreads\(\)", s)]
    assert sync and fence, "no fence before the refill"
    used = [k for k, s in enumerate(code) if re.search(r"\bslot\b|\bsrow\b|transform\(", s)]
    stored = any("transform(" in s for s in code)  # the transform works in the slot
    if stored:
        assert max(used) < fence[-1] < sync[-1], "stores must be fenced before the barrier"
    else:
        assert max(used) < fence[-1]
