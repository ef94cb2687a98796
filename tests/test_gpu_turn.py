"""The corner turn between the compressions, at tile edges: turned output and input equal the dense form turned by torch,
bit for bit (the turn only moves values)."""

import pytest

from paper_2605_28451_gb300 import bfpfft as B
from paper_2605_28451_gb300 import build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib(cuda_ready):
    build.build()
    B.lib()


def noise(shape, storage, seed):
    import torch
    x = torch.randn(shape + (2,), device="cuda:0", generator=torch.Generator(device="cuda:0").manual_seed(seed))
    return x.half() if storage == B.F16_BFP else torch.view_as_complex(x)


# lines whose points are turned; 63 ... 66 and 31 ... 34 are the edges of a tile of either type, 2400 takes several tiles
# per CTA
@pytest.mark.parametrize("lines", [1, 2, 31, 34, 63, 64, 65, 66, 100, 129, 1001, 2400])
@pytest.mark.parametrize("n", [256, 4096])
@pytest.mark.parametrize("storage", [B.F16_BFP, B.F32])
def test_turned_and_dense_agree(lines, n, storage):
    import torch
    x = noise((lines, n), storage, lines)
    h = noise((n,), B.F32, 7) / n ** 0.5
    dense, turned = torch.zeros_like(x), torch.zeros_like(x).reshape((n, lines) + x.shape[2:])
    B.sar_range_compress(x, storage, dense, storage, h, lines, n, False)
    B.sar_range_compress(x, storage, turned, storage, h, lines, n, True)
    torch.cuda.synchronize()
    assert torch.equal(turned, dense.transpose(0, 1))
    # the azimuth call turns its input (layout 0) and its output, n pulses by `lines` range bins
    a, b = torch.zeros_like(turned), torch.zeros_like(turned)
    B.sar_azimuth_compress(x.transpose(0, 1).contiguous(), storage, 0, a, storage, h, n, lines)
    B.sar_azimuth_compress(x, storage, 1, b, storage, h, n, lines)
    torch.cuda.synchronize()
    assert torch.equal(a, turned) and torch.equal(b, turned)
    assert B.bfpfft_device_status() == B.OK
