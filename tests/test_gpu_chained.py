"""Kernels whose CTAs start under the tail of the stream's previous kernel: chains in which every kernel reads what the
one before has just written, small enough that all their CTAs fit on the GPU together, give bit for bit what the same
calls give with a synchronisation after each; on a stream, and captured between a memset, a copy and a fork.
"""

import pytest

from paper_2605_28451_gb300 import bfpfft as B
from paper_2605_28451_gb300 import build, synth

pytestmark = pytest.mark.gpu

STEPS = 12


@pytest.fixture(scope="module", autouse=True)
def _lib(cuda_ready):
    build.build()
    B.lib()


def noise(shape, seed):
    import torch
    return torch.randn(shape, device="cuda:0", generator=torch.Generator(device="cuda:0").manual_seed(seed))


def run_chain(plans, bufs, between):
    """Transforms there and back through three buffers, with a torch kernel in the chain's middle."""
    import torch
    for k in range(STEPS):
        B.bfpfft_exec(plans[k % 2], bufs[k % 3], bufs[(k + 1) % 3])
        if k == STEPS // 2:
            bufs[(k + 1) % 3].mul_(0.5)
        if between:
            torch.cuda.synchronize()
    return bufs[STEPS % 3]


def run_captured(body, reset):
    """body() in a graph, behind a memset and a copy and beside a forked stream; replayed twice."""
    import torch
    stream, side, graph = torch.cuda.Stream(), torch.cuda.Stream(), torch.cuda.CUDAGraph()
    reset()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        body()
    torch.cuda.synchronize()
    reset()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=stream):
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            torch.ones(8, device="cuda:0").mul_(2)
        reset()
        out = body()
        torch.cuda.current_stream().wait_stream(side)
    graph.replay()
    graph.replay()
    torch.cuda.synchronize()
    return out.clone()


# n, lines: each kernel of the row family at a batch that leaves the GPU partly idle
SHAPES = [(16, 40), (256, 8), (512, 300), (1024, 77), (2048, 1300), (4096, 100), (4096, 1900), (8192, 60), (16384, 9),
          (16384, 200), (32768, 3), (65536, 12)]


@pytest.mark.parametrize("n,lines", SHAPES)
@pytest.mark.parametrize("storage,arith", [(B.F16_BFP, None), (B.F32, None), (B.F16_BFP, "tc"), (B.F16_BFP, "f16"),
                                           (B.BF16, None), (B.F16_BFP, "tma")])
def test_dependent_transforms(n, lines, storage, arith, monkeypatch):
    import torch
    if arith == "tc" and n != 4096:
        pytest.skip("4096 points only")
    if n > 16384 and (arith == "f16" or storage == B.BF16):
        pytest.skip("16-bit arithmetic up to 16384 points")
    if arith == "tma":
        monkeypatch.setenv("BFPFFT_ROWS", "tma")
    start = noise((lines, n, 2), n + lines)
    start = {B.F16_BFP: start.half(), B.BF16: start.bfloat16()}.get(storage, torch.view_as_complex(start))
    plans = [B.bfpfft_plan_create(n, lines, storage, d) for d in (B.FORWARD, B.INVERSE)]
    for p in plans if arith in ("tc", "f16") else ():
        B.bfpfft_plan_set_arith(p, B.ARITH_F16 if arith == "f16" else B.ARITH_F16_MUL_F32_ACC)

    def bufs():
        return [start.clone(), torch.zeros_like(start), torch.zeros_like(start)]

    expect = run_chain(plans, bufs(), True).clone()
    torch.cuda.synchronize()
    for _ in range(3):
        assert torch.equal(run_chain(plans, bufs(), False), expect)
    own = bufs()

    def reset():
        own[0].copy_(start)
        own[1].zero_()
        own[2].zero_()

    assert torch.equal(run_captured(lambda: run_chain(plans, own, False), reset), expect)
    for p in plans:
        assert B.bfpfft_plan_status(p) == B.OK


@pytest.mark.parametrize("count", [40, 1500])
@pytest.mark.parametrize("storage", [B.F16_BFP, B.F32])
@pytest.mark.parametrize("flags", [0, B.MANY_PER_LENGTH])
def test_dependent_ragged_batches(count, storage, flags):
    """The persistent kernel, or per-length kernels on the caller's stream and the plan's own, each exec reading what the
    last one wrote."""
    import torch
    n = synth.uneven_lengths(count, seed=count)
    off = n.cumsum() - n
    start = noise((int(n.sum()), 2), count)
    start = start.half() if storage == B.F16_BFP else torch.view_as_complex(start)
    plans = [B.bfpfft_plan_create_many(n, off, storage, d) for d in (B.FORWARD, B.INVERSE)]
    for p in plans:
        B.bfpfft_plan_set_many_schedule(p, 0, flags)
    own = [start.clone(), torch.zeros_like(start), torch.zeros_like(start)]

    def reset():
        own[0].copy_(start)
        own[1].zero_()
        own[2].zero_()

    expect = run_chain(plans, own, True).clone()
    for _ in range(3):
        reset()
        assert torch.equal(run_chain(plans, own, False), expect)
    assert torch.equal(run_captured(lambda: run_chain(plans, own, False), reset), expect)
    for p in plans:
        assert B.bfpfft_plan_status(p) == B.OK


@pytest.mark.parametrize("n,lines", [(256, 30), (4096, 200), (16384, 40)])
def test_adaptive_exponents_in_one_chain(n, lines):
    """Mantissas and exponents written by one kernel are the next one's input."""
    import torch
    start = noise((lines, n, 2), n).half()
    plans = [B.bfpfft_plan_create(n, lines, B.F16_ADAPTIVE, d) for d in (B.FORWARD, B.INVERSE)]
    results = []
    for between in (True, False, False):
        x = [start.clone(), torch.zeros_like(start)]
        e = [torch.full((lines,), 3, dtype=torch.int32, device="cuda:0"), torch.zeros(lines, dtype=torch.int32,
                                                                                      device="cuda:0")]
        for k in range(STEPS):
            B.bfpfft_exec_adaptive(plans[k % 2], x[k % 2], e[k % 2], x[(k + 1) % 2], e[(k + 1) % 2])
            if between:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        results.append((x[0], e[0]))
    for x, e in results[1:]:
        assert torch.equal(x, results[0][0]) and torch.equal(e, results[0][1])


@pytest.mark.parametrize("n_az,n_rg", [(512, 256), (256, 1024), (1024, 2048)])
@pytest.mark.parametrize("out", [B.F16_BFP, B.F32])
def test_filter_made_and_used_in_one_chain(n_az, n_rg, out):
    """A spectrum computed by one kernel is the next one's filter; then range, turn, azimuth and the RDA lines."""
    import torch
    raw = torch.view_as_complex(noise((n_az, n_rg, 2), 5))
    pulse = torch.view_as_complex(noise((1, n_rg, 2), 6)) / n_rg ** 0.5
    geo = synth.radar_geometry(1024)
    geo = (geo.range_cell_m, geo.prf_hz, geo.wavelength_m, geo.speed_mps, geo.centre_range_m)
    plan = B.bfpfft_plan_create(n_rg, 1, B.F32, B.FORWARD)
    h = torch.zeros((1, n_rg), dtype=torch.complex64, device="cuda:0")

    def empty(shape):
        if out == B.F16_BFP:
            return torch.zeros(shape + (2,), dtype=torch.float16, device="cuda:0")
        return torch.zeros(shape, dtype=torch.complex64, device="cuda:0")

    kept = empty((n_az, n_rg)), empty((n_rg, n_az)), empty((n_az, n_rg))
    both = torch.zeros((2,) + tuple(kept[0].shape), dtype=kept[0].dtype, device="cuda:0")

    def reset():
        h.zero_()
        for x in kept:
            x.zero_()

    def body(between=False):
        filtered, rc, img = kept
        wait = torch.cuda.synchronize if between else (lambda: None)
        B.bfpfft_exec(plan, pulse, h)
        wait()
        B.bfp_spectral_filter(raw, B.F32, h, 0, filtered, out, n_rg, n_az)
        wait()
        B.sar_range_compress(raw, B.F32, rc, out, h, n_az, n_rg, True)
        wait()
        B.sar_rda_image(raw, B.F32, img, out, h, n_az, n_rg, geo, n_az // 2,
                        B.RDA_RCMC | B.RDA_RANGE_DEPENDENT | B.RDA_PEAK_NORMALISE)
        wait()
        both[0].copy_(filtered)
        both[1].copy_(rc.reshape(both[1].shape))
        both[1].add_(img)
        return both

    reset()
    expect = body(True).clone()
    assert torch.isfinite(torch.view_as_real(expect) if expect.is_complex() else expect).all()
    for _ in range(3):
        reset()
        assert torch.equal(body(), expect)
    assert torch.equal(run_captured(body, reset), expect)
    assert B.bfpfft_device_status() == B.OK
