"""The RCMC and azimuth-filter lines at every line length of their range (256 ... 8192), short and long apertures and a
geometry whose migration runs over many cells, against the FP64 oracle on noise-like echoes.  Bars as in
tests/test_gpu_rda.py: FP32 relative L2 <= 1e-5, FP16 image SQNR >= 40 dB.
"""

import numpy as np
import pytest

from oracle import metrics, rda
from paper_2605_28451_gb300 import bfpfft as B
from paper_2605_28451_gb300 import build, synth

from _helpers import empty_like_storage, from_device, storage_round, to_device

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib(cuda_ready):
    build.build()
    B.lib()


def geometry(wide):
    geo = synth.radar_geometry(1024)
    if wide:                       # three times the wavelength: up to 20 cells of migration at the band's edge
        geo.wavelength_m *= 1.5
        geo.range_cell_m *= 0.25
    return geo


@pytest.mark.parametrize("n_az,n_rg,aperture", [(256, 256, 2), (256, 512, 256), (512, 256, 100), (512, 2048, 512),
                                                (1024, 256, 1024), (256, 8192, 128), (8192, 256, 4096),
                                                (2048, 512, 700)])
@pytest.mark.parametrize("wide", [False, True])
@pytest.mark.parametrize("dtype", [B.F32, B.F16_BFP])
def test_line_lengths(n_az, n_rg, aperture, wide, dtype):
    import torch
    geo = geometry(wide)
    raw = storage_round(synth.complex_gaussian(n_az, n_rg, seed=n_az + n_rg), B.F32)
    pulse = synth.complex_gaussian(1, n_rg, seed=3)[0] / np.sqrt(n_rg)
    hr = storage_round(np.conj(np.fft.fft(pulse)), B.F32)
    flags = B.RDA_RCMC | B.RDA_RANGE_DEPENDENT | B.RDA_PEAK_NORMALISE
    img = empty_like_storage((n_az, n_rg), dtype)
    B.sar_rda_image(to_device(raw, B.F32), B.F32, img, dtype, to_device(hr, B.F32), n_az, n_rg,
                    (geo.range_cell_m, geo.prf_hz, geo.wavelength_m, geo.speed_mps, geo.centre_range_m), aperture,
                    flags)
    torch.cuda.synchronize()
    assert B.bfpfft_device_status() == B.OK
    expect = rda.image(raw, hr, geo, aperture, True, True, True)
    got = from_device(img, dtype)
    if dtype == B.F32:
        assert metrics.rel_l2(expect, got) <= 1e-5
    else:
        assert metrics.sqnr_db(expect, got) >= 40.0
