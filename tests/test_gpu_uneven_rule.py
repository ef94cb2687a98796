"""The schedule an untuned uneven plan takes by its lengths: the persistent kernel where many lengths share the points
(a launch each costs more than the dense kernels save), one launch per length where few do.  The schedules' kernels
round differently, so the bits tell them apart."""

import numpy as np
import pytest

from paper_2605_28451_gb300 import bfpfft as B
from paper_2605_28451_gb300 import build

pytestmark = pytest.mark.gpu

ALL = range(4, 17)
MIXES = [   # log2 lengths, log2 points in all, one launch per length
    ([10], 22, False),
    ([10], 23, True),
    ([12], 23, True),
    ([8, 9, 10], 23, True),
    ([8, 16], 23, True),
    (range(6, 11), 23, False),
    (range(6, 11), 24, True),
    (range(4, 13), 24, False),
    (range(4, 13), 25, True),
    (ALL, 23, False),
    (ALL, 24, False),
    (ALL, 25, True),
]


@pytest.mark.parametrize("logs,log_points,per_length", MIXES)
def test_schedule_by_lengths(cuda_ready, logs, log_points, per_length):
    import torch
    build.build()
    logs = list(logs)
    n = np.concatenate([np.full(((1 << log_points) // len(logs) >> l) + 1, 1 << l, dtype=np.int64) for l in logs])
    if log_points == 22:
        n = n[:-1]
    np.random.default_rng(0).shuffle(n)
    plan = B.bfpfft_plan_create_many(n, np.cumsum(n) - n, B.F16_BFP, B.FORWARD)
    g = torch.Generator(device="cuda:0").manual_seed(log_points)
    x = torch.randn((int(n.sum()), 2), device="cuda:0", generator=g).half()
    default, persistent, listed = (torch.empty_like(x) for _ in range(3))
    B.bfpfft_exec(plan, x, default)
    B.bfpfft_plan_set_many_schedule(plan, 0, 0)
    B.bfpfft_exec(plan, x, persistent)
    B.bfpfft_plan_set_many_schedule(plan, 0, B.MANY_PER_LENGTH)
    B.bfpfft_exec(plan, x, listed)
    torch.cuda.synchronize()
    assert not torch.equal(persistent, listed)
    assert torch.equal(default, listed if per_length else persistent)
    assert B.bfpfft_plan_status(plan) == B.OK
