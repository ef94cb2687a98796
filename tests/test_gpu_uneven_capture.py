"""One uneven plan executed on a stream while another stream's capture of it is still open, both ways a capture comes
about: the caller's own, and another thread's.  Long and short lines together, so that the per-length schedule has both."""

import threading

import numpy as np
import pytest

from paper_2605_28451_gb300 import bfpfft as B
from paper_2605_28451_gb300 import build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib(cuda_ready):
    build.build()
    B.lib()


def plan_and_data():
    import torch
    n = np.array([65536, 32768, 4096, 4096, 256, 16, 1024] * 3, dtype=np.int64)
    plan = B.bfpfft_plan_create_many(n, np.cumsum(n) - n, B.F16_BFP, B.FORWARD)
    B.bfpfft_plan_set_many_schedule(plan, 0, B.MANY_PER_LENGTH)
    g = torch.Generator(device="cuda:0").manual_seed(3)
    xs = [torch.randn((int(n.sum()), 2), device="cuda:0", generator=g).half() for _ in range(2)]
    expect = [torch.empty_like(x) for x in xs]
    for x, y in zip(xs, expect):
        B.bfpfft_exec(plan, x, y)
    torch.cuda.synchronize()
    return plan, xs, expect


@pytest.mark.parametrize("threads", [1, 2])
def test_executed_while_captured(threads):
    import torch
    plan, xs, expect = plan_and_data()
    captured, eager = torch.zeros_like(xs[0]), torch.zeros_like(xs[1])
    capturing, other, graph = torch.cuda.Stream(), torch.cuda.Stream(), torch.cuda.CUDAGraph()

    def execute():
        B.bfpfft_exec(plan, xs[1], eager, stream=other)
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=capturing, capture_error_mode="thread_local"):
        B.bfpfft_exec(plan, xs[0], captured)
        if threads == 1:
            execute()
        else:
            t = threading.Thread(target=execute)
            t.start()
            t.join()
        B.bfpfft_exec(plan, captured, captured)
    other.synchronize()
    assert torch.equal(eager, expect[1])
    for _ in range(2):
        graph.replay()
    torch.cuda.synchronize()
    twice = torch.empty_like(xs[0])
    B.bfpfft_exec(plan, expect[0], twice)
    torch.cuda.synchronize()
    assert torch.equal(captured, twice)
    assert B.bfpfft_plan_status(plan) == B.OK


def test_two_captures_open_at_once():
    """Each capture forks onto a stream of its own; an execution after both takes either again."""
    import torch
    plan, xs, expect = plan_and_data()
    outs, graphs = [torch.zeros_like(x) for x in xs], [torch.cuda.CUDAGraph() for _ in xs]
    first, second = torch.cuda.Stream(), torch.cuda.Stream()
    opened, done = threading.Event(), threading.Event()

    def hold_open():
        with torch.cuda.graph(graphs[1], stream=second, capture_error_mode="thread_local"):
            B.bfpfft_exec(plan, xs[1], outs[1])
            opened.set()
            done.wait(60)
            B.bfpfft_exec(plan, xs[1], outs[1])
    torch.cuda.synchronize()
    t = threading.Thread(target=hold_open)
    t.start()
    assert opened.wait(60)
    B.bfpfft_exec_graph(plan, xs[0], outs[0], stream=first)      # captures by itself, then replays
    done.set()
    t.join()
    graphs[1].replay()
    torch.cuda.synchronize()
    assert torch.equal(outs[0], expect[0]) and torch.equal(outs[1], expect[1])
    eager = torch.zeros_like(xs[0])
    B.bfpfft_exec(plan, xs[0], eager)
    torch.cuda.synchronize()
    assert torch.equal(eager, expect[0])
    assert B.bfpfft_plan_status(plan) == B.OK
