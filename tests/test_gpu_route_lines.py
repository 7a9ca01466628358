"""Kernels of two tile widths give the same bits on either side of the line between them."""

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rosar():
    from paper_2309_08038_gb300 import build
    build.build()
    import paper_2309_08038_gb300 as r
    return r


def _c(rng, *shape):
    return (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)).astype(np.complex64)


# 1024 samples: tiles of 4 pulses where the fullest SM holds an odd number of them (up to 608 pulses, 1217 to 1824) or the
# row stride is odd, else of 8; a stack of two scans counts twice, so that it takes the other width
@pytest.mark.parametrize("n_az", [2, 304, 606, 608, 610, 1216, 1218, 1217, 1820])
def test_range_compression_of_1024_samples(rosar, n_az):
    import torch
    rng = np.random.default_rng(n_az)
    raw = torch.from_numpy(_c(rng, 3, n_az, 1024)).cuda()
    win = torch.from_numpy(synth.hann_window(1024)).cuda()
    one = torch.stack([rosar.range_compress(r, win) for r in raw])
    assert torch.equal(rosar.range_compress(raw, win), one)
    assert torch.equal(rosar.range_compress(raw[:2], win), one[:2])
    ref = torch.fft.fft(raw[0].cdouble() * win.double(), dim=-1)
    l = torch.arange(1024, dtype=torch.float64, device="cuda")
    ref = (ref * torch.polar(torch.ones_like(l), torch.pi * torch.remainder(l * 1023 / 1024, 2.0))).T
    assert torch.linalg.norm(one[0] - ref) <= 2e-6 * torch.linalg.norm(ref)       # the range FFT's bar
