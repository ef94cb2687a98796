"""A matched filter has the same bits whichever row kernels a batch of its length runs on: those of the 16-point kernel
(and of the four-step kernel from 32768 points on)."""

import pytest

from paper_2605_28451_gb300 import bfpfft as B
from paper_2605_28451_gb300 import build

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("log2n", range(4, 17))
@pytest.mark.parametrize("peak", [False, True])
def test_filter_is_that_of_the_general_kernel(cuda_ready, monkeypatch, log2n, peak):
    import torch
    build.build()
    n = 1 << log2n
    g = torch.Generator(device="cuda:0").manual_seed(n)
    ref = torch.view_as_complex(torch.randn((n, 2), device="cuda:0", generator=g))
    default, general = torch.empty_like(ref), torch.empty_like(ref)
    B.sar_make_filter(ref, n, peak, default)
    monkeypatch.setenv("BFPFFT_ROWS", "plain")
    B.sar_make_filter(ref, n, peak, general)
    torch.cuda.synchronize()
    assert torch.equal(torch.view_as_real(default), torch.view_as_real(general))
