"""The shared-memory transforms at every length: spectra of random cubes against torch's FP64 FFT.

Tolerance: radix-2 stages in FP32 with correctly rounded twiddles add at most about 1.2e-7 rms
per stage in quadrature; 12 + 9 stages give 5.5e-7, bounded here by 1e-6 relative L2."""
import pytest
import torch

from sbr_inputs import CfarParams, radar_single_tx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ns,nc", [(n, c) for n in (32, 64, 128, 256, 512, 1024, 2048, 4096)
                                   for c in (1, 2, 8, 16, 128, 512) if n * c <= 1 << 17])
def test_spectrum(sbr, ns, nc):
    radar = radar_single_tx(ns, nc)
    cube = torch.randn(4, nc, ns, 2, generator=torch.Generator(device="cuda").manual_seed(ns + nc), device="cuda")
    state = sbr.power_map(cube, radar, CfarParams())
    ref = torch.fft.fft(torch.fft.fft(torch.view_as_complex(cube.double()), dim=2), dim=1)
    got = torch.view_as_complex(state.spectrum().double())
    assert float((got - ref).norm() / ref.norm()) <= 1e-6
