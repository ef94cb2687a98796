"""GPU parity of the kernels with 32 or 64 points per thread (lines of 512 ... 16384 points) where they can go
wrong: batches that leave a CTA's last lines empty, batches on either side of the line counts from which 2048 and
4096 points take them, the persistent CTAs of 16384 points walking several lines, in-place calls, host buffers and
listed lines.  Bars are those of tests/test_gpu_fft.py: FP32 relative L2 <= 1e-6, FP16 within half an ulp plus the
FP32 arithmetic, FP8 the oracle's rounding or one step across a boundary.
"""

import numpy as np
import pytest

from oracle import fft as F
from oracle import metrics
from paper_2605_28451_gb300 import bfpfft as B
from paper_2605_28451_gb300 import build

from _helpers import fp8_close, fp16_elementwise_ok, from_device

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib(cuda_ready):
    build.build()
    B.lib()


def lines(batch, n, dtype, seed):
    import torch
    g = torch.Generator(device="cuda:0").manual_seed(seed)
    x = torch.randn((batch, n, 2), device="cuda:0", generator=g)
    if dtype == B.F32:
        return torch.view_as_complex(x)
    return x.to(torch.float16) if dtype == B.F16_BFP else x.to(torch.float8_e4m3fn).view(torch.uint8)


def check(got, exact, dtype):
    if dtype == B.F32:
        assert metrics.rel_l2(exact, got) <= 1e-6
    elif dtype == B.F16_BFP:
        ok, worst = fp16_elementwise_ok(got, exact)
        assert ok, worst
    else:
        fp8_close(got, exact, "e4m3")


EDGES = [(512, 1), (512, 5), (512, 3001), (1024, 1), (1024, 3), (1024, 2049), (2048, 1215), (2048, 1216), (2048, 1217),
         (4096, 1823), (4096, 1824), (4096, 1825), (8192, 1), (8192, 306), (16384, 1), (16384, 153), (16384, 307)]


@pytest.mark.parametrize("n,batch", EDGES)
@pytest.mark.parametrize("dtype", [B.F16_BFP, B.F32, B.E4M3_BFP])
@pytest.mark.parametrize("direction", [B.FORWARD, B.INVERSE])
def test_edges_of_the_batch(n, batch, dtype, direction):
    import torch
    plan = B.bfpfft_plan_create(n, batch, dtype, direction)
    x = lines(batch, n, dtype, n + batch)
    y = torch.empty_like(x)
    B.bfpfft_exec(plan, x, y)
    z = x.clone()
    B.bfpfft_exec(plan, z, z)
    torch.cuda.synchronize()
    assert torch.equal(y.view(torch.uint8) if dtype != B.F32 else torch.view_as_real(y),
                       z.view(torch.uint8) if dtype != B.F32 else torch.view_as_real(z))
    assert B.bfpfft_plan_status(plan) == B.OK
    some = sorted({0, 1 % batch, batch // 2, max(0, batch - 2), batch - 1})
    e_in, e_out = B.bfpfft_plan_scale_exp(plan)
    v = from_device(x[some], dtype) * 2.0 ** e_in
    exact = (F.fft(v) if direction == B.FORWARD else F.ifft(v)) * 2.0 ** -e_out
    check(from_device(y[some], dtype), exact, dtype)


@pytest.mark.parametrize("n,batch", [(512, 9), (2048, 1217), (4096, 1825), (16384, 200)])
def test_host_buffer_and_listed_lines_give_the_same_bits(n, batch):
    import torch
    x = lines(batch, n, B.F16_BFP, 7 * n)
    y = torch.empty_like(x)
    plan = B.bfpfft_plan_create(n, batch, B.F16_BFP, B.FORWARD)
    B.bfpfft_exec(plan, x, y)
    host = x.cpu().pin_memory()
    from_host = torch.empty_like(x)
    B.bfpfft_exec(plan, host, from_host)
    pitch = n + 16                                        # lines with a gap, in reverse order
    offsets = (np.arange(batch)[::-1] * pitch).copy()
    packed = torch.zeros((batch * pitch, 2), dtype=torch.float16, device="cuda:0")
    packed.view(batch, pitch, 2)[:, :n] = x.flip(0)
    out = torch.zeros_like(packed)
    many = B.bfpfft_plan_create_many(np.full(batch, n), offsets, B.F16_BFP, B.FORWARD)
    B.bfpfft_plan_set_many_schedule(many, 0, B.MANY_PER_LENGTH)
    B.bfpfft_exec(many, packed, out)
    torch.cuda.synchronize()
    assert torch.equal(y, from_host)
    assert torch.equal(out.view(batch, pitch, 2)[:, :n].flip(0), y)
    assert B.bfpfft_plan_status(plan) == B.OK and B.bfpfft_plan_status(many) == B.OK


@pytest.mark.parametrize("n", [512, 1024, 8192, 16384])
@pytest.mark.parametrize("batch", [1, 5, 611])
@pytest.mark.parametrize("x_dtype,out_dtype", [(B.F16_BFP, B.F16_BFP), (B.F32, B.F16_BFP), (B.F32, B.F32), (B.F16_BFP, B.F32)])
def test_filtered_lines(n, batch, x_dtype, out_dtype):
    import torch
    x = lines(batch, n, x_dtype, 11 * n + batch)
    h = lines(batch, n, B.F32, 13 * n + batch)
    y = torch.empty((batch, n), dtype=torch.complex64, device="cuda:0") if out_dtype == B.F32 else \
        torch.empty((batch, n, 2), dtype=torch.float16, device="cuda:0")
    some = sorted({0, batch // 2, batch - 1})
    for stride in (0, n):
        B.bfp_spectral_filter(x, x_dtype, h, stride, y, out_dtype, n, batch)
        torch.cuda.synchronize()
        hs = from_device(h[some] if stride else h[:1], B.F32)
        check(from_device(y[some], out_dtype), F.ifft(F.fft(from_device(x[some], x_dtype)) * hs), out_dtype)
    assert B.bfpfft_device_status() == B.OK
