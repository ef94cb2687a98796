"""The scratch that a gradient call left with the library's pool goes back to the driver when asked."""

import pytest

from paper_2605_28451_gb300 import autofocus as GA
from paper_2605_28451_gb300 import bfpfft as B
from paper_2605_28451_gb300 import build

pytestmark = pytest.mark.gpu


def test_scratch_is_given_back(cuda_ready):
    import torch
    build.build()
    n_az, n_rg = 4096, 8192                                  # an image of 256 MiB
    rc = torch.randn((n_rg, n_az, 2), device="cuda:0").half()
    ha = torch.ones(n_az, dtype=torch.complex64, device="cuda:0")
    phi, grad, again = (torch.zeros(n_az, device="cuda:0") for _ in range(3))
    ws = GA.Workspace(n_az, "cuda:0")

    def step(out):
        B.sar_autofocus_grad(rc, B.F16_BFP, phi, ha, n_az, n_rg, out, ws.stats, ws.buf, ws.bytes)
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]
    B.bfpfft_release_scratch()
    free = step(grad)
    B.bfpfft_release_scratch()
    B.bfpfft_release_scratch()                               # nothing left to give: no error
    assert torch.cuda.mem_get_info()[0] - free >= n_az * n_rg * 8
    step(again)
    assert torch.equal(grad, again)
