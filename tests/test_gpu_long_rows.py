"""GPU parity of the cluster kernel for lines of 32768 and 65536 points (long_rows.cuh) on either side of the batch
from which it takes over the four-step kernel, in every storage type and direction, in place, from host buffers, on
listed lines and with the row exchange in FP16 words.  Bars as in tests/test_gpu_fft.py; the FP16 row exchange is one
more FP16 storage point (6 * 2^-11 rms per element, 55 dB).
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
    if dtype == B.F16_BFP:
        return x.to(torch.float16)
    return x.to(torch.float8_e4m3fn if dtype == B.E4M3_BFP else torch.float8_e5m2).view(torch.uint8)


def expect(x, plan, direction, dtype):
    e_in, e_out = B.bfpfft_plan_scale_exp(plan)
    v = from_device(x, dtype) * 2.0 ** e_in
    return (F.fft(v) if direction == B.FORWARD else F.ifft(v)) * 2.0 ** -e_out


@pytest.mark.parametrize("n,batch", [(65536, 9), (65536, 10), (65536, 61), (32768, 19), (32768, 20), (32768, 117)])
@pytest.mark.parametrize("dtype", [B.F16_BFP, B.F32, B.E4M3_BFP, B.E5M2_BFP])
@pytest.mark.parametrize("direction", [B.FORWARD, B.INVERSE])
def test_around_the_switch(n, batch, dtype, direction):
    import torch
    plan = B.bfpfft_plan_create(n, batch, dtype, direction)
    x = lines(batch, n, dtype, n + batch)
    y = torch.empty_like(x)
    B.bfpfft_exec(plan, x, y)
    z = x.clone()
    B.bfpfft_exec(plan, z, z)
    torch.cuda.synchronize()
    assert torch.equal(torch.view_as_real(y) if dtype == B.F32 else y, torch.view_as_real(z) if dtype == B.F32 else z)
    assert B.bfpfft_plan_status(plan) == B.OK
    some = [0, batch // 2, batch - 1]
    exact, got = expect(x[some], plan, direction, dtype), from_device(y[some], dtype)
    if dtype == B.F32:
        assert metrics.rel_l2(exact, got) <= 1e-6
    elif dtype == B.F16_BFP:
        ok, worst = fp16_elementwise_ok(got, exact)
        assert ok, worst
    else:
        fp8_close(got, exact, "e4m3" if dtype == B.E4M3_BFP else "e5m2")


@pytest.mark.parametrize("n,batch", [(65536, 11), (32768, 21)])
@pytest.mark.parametrize("direction", [B.FORWARD, B.INVERSE])
def test_fp16_row_exchange(n, batch, direction, monkeypatch):
    import torch
    monkeypatch.setenv("BFPFFT_ROWS", "h16_l2")
    plan = B.bfpfft_plan_create(n, batch, B.F16_BFP, direction)
    x = lines(batch, n, B.F16_BFP, 3 * n)
    y = torch.empty_like(x)
    B.bfpfft_exec(plan, x, y)
    torch.cuda.synchronize()
    assert B.bfpfft_plan_status(plan) == B.OK
    exact, got = expect(x[[0, batch - 1]], plan, direction, B.F16_BFP), from_device(y[[0, batch - 1]], B.F16_BFP)
    bound = 2.0 ** -11 * (np.abs(exact) + 6.0 * np.sqrt(np.mean(np.abs(exact) ** 2)))
    assert np.all(np.abs(got.real - exact.real) <= bound) and np.all(np.abs(got.imag - exact.imag) <= bound)
    assert metrics.sqnr_db(exact, got) >= 55.0


@pytest.mark.parametrize("n,batch", [(65536, 11), (32768, 23)])
def test_host_buffer_listed_lines_and_finite_check(n, batch):
    import torch
    x = lines(batch, n, B.F16_BFP, 5 * n)
    y = torch.empty_like(x)
    plan = B.bfpfft_plan_create(n, batch, B.F16_BFP, B.FORWARD)
    B.bfpfft_plan_set_flags(plan, B.CHECK_FINITE)
    B.bfpfft_exec(plan, x, y)
    from_host = torch.empty_like(x)
    B.bfpfft_exec(plan, x.cpu().pin_memory(), from_host)
    pitch = n + 32
    packed = torch.zeros((batch * pitch, 2), dtype=torch.float16, device="cuda:0")
    packed.view(batch, pitch, 2)[:, :n] = x.flip(0)
    out = torch.zeros_like(packed)
    many = B.bfpfft_plan_create_many(np.full(batch, n), (np.arange(batch)[::-1] * pitch).copy(), B.F16_BFP, B.FORWARD)
    B.bfpfft_plan_set_many_schedule(many, 0, B.MANY_PER_LENGTH)
    B.bfpfft_exec(many, packed, out)
    torch.cuda.synchronize()
    assert torch.equal(y, from_host)
    assert torch.equal(out.view(batch, pitch, 2)[:, :n].flip(0), y)
    assert B.bfpfft_plan_status(plan) == B.OK
    x[batch - 1, 5, 0] = float("inf")
    B.bfpfft_exec(plan, x, y)
    torch.cuda.synchronize()
    assert B.bfpfft_plan_status(plan) == B.ERR_NONFINITE
