"""The centring factors of the range adjoint, bin by bin: a gradient of one bin a pulse, with and without them."""

import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# Two table entries, each component rounded once or twice (2^-24 of it), their product and its product with the bin: at
# most 2.5e-7 of a factor; the transforms' own rounding is the same in both runs and the rest averages out over L samples.
TOL_FACTOR = 2.5e-7


@pytest.fixture(scope="module")
def rosar():
    from paper_2309_08038_gb300 import build
    build.build()
    import paper_2309_08038_gb300 as r
    return r


@pytest.mark.parametrize("L", [8, 16, 32, 64, 128, 256, 512, 1024, 2048, 4096])
def test_centring_factors(rosar, L):
    import torch
    g = torch.eye(L, dtype=torch.complex64, device="cuda")            # pulse n has bin n alone
    got = rosar.range_compress_adjoint(g, None, centred=True).cpu().numpy().astype(np.complex128)
    plain = rosar.range_compress_adjoint(g, None, centred=False).cpu().numpy().astype(np.complex128)
    factor = (got * plain.conj()).sum(1) / (np.abs(plain) ** 2).sum(1)
    l = np.arange(L, dtype=np.float64)
    want = np.exp(-1j * math.pi * np.remainder(l * (L - 1) / L, 2.0))          # the conjugate of c_l
    assert np.abs(factor - want).max() <= TOL_FACTOR
