"""The schedule an untuned uneven plan takes by its size, and one plan used by two host threads on two streams."""

import threading

import numpy as np
import pytest

from paper_2605_28451_gb300 import bfpfft as B
from paper_2605_28451_gb300 import build

pytestmark = pytest.mark.gpu

LARGE = 1 << 23


@pytest.fixture(scope="module", autouse=True)
def _lib(cuda_ready):
    build.build()
    B.lib()


def batch(points, seed):
    """Lengths 16 ... 65536 in mixed order that add up to `points`, and their data."""
    import torch
    rng = np.random.default_rng(seed)
    lengths, left = [], points
    while left:
        n = min(1 << int(rng.integers(4, 17)), 1 << (left.bit_length() - 1))
        lengths.append(n)
        left -= n
    n = np.array(lengths, dtype=np.int64)
    x = torch.randn((points, 2), device="cuda:0", generator=torch.Generator(device="cuda:0").manual_seed(seed)).half()
    return n, np.cumsum(n) - n, x


@pytest.mark.parametrize("points,flags", [(LARGE - 16, 0), (LARGE, B.MANY_PER_LENGTH), (LARGE + 48, B.MANY_PER_LENGTH)])
@pytest.mark.parametrize("direction", [B.FORWARD, B.INVERSE])
def test_schedule_by_size(points, flags, direction):
    import torch
    n, off, x = batch(points, points)
    plan = B.bfpfft_plan_create_many(n, off, B.F16_BFP, direction)
    y, z = torch.empty_like(x), torch.empty_like(x)
    B.bfpfft_exec(plan, x, y)
    B.bfpfft_plan_set_many_schedule(plan, 0, flags)
    B.bfpfft_exec(plan, x, z)
    torch.cuda.synchronize()
    assert torch.equal(y, z)
    assert B.bfpfft_plan_status(plan) == B.OK


def test_two_threads_share_a_large_plan():
    import torch
    n, off, x = batch(LARGE, 1)
    plan = B.bfpfft_plan_create_many(n, off, B.F16_BFP, B.FORWARD)
    expect = torch.empty_like(x)
    B.bfpfft_exec(plan, x, expect)
    torch.cuda.synchronize()
    outs = [torch.zeros_like(x) for _ in range(2)]

    def work(k):
        stream = torch.cuda.Stream()
        mine = torch.zeros_like(x)
        torch.cuda.synchronize()
        with torch.cuda.stream(stream):
            for _ in range(20):
                mine.copy_(x)                      # the short lengths' stream has to wait for this copy
                B.bfpfft_exec(plan, mine, outs[k])
                mine.zero_()                       # ... and this fill for the short lengths
        stream.synchronize()
    threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert torch.equal(outs[0], expect) and torch.equal(outs[1], expect)
