"""The weight gradient from stored spectra, for every order in which the row filter stores them: each compile-time length
with few and with many rows, and run-time lengths."""

import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rosar():
    from paper_2309_08038_gb300 import build
    build.build()
    import paper_2309_08038_gb300 as r
    return r


def _c(rng, *shape):
    return (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)).astype(np.complex64)


# 10 rows in one call, and just above the lines between the variants (152 and 304 rows)
@pytest.mark.parametrize("n_az,n_scans", [(14400, 2), (14400, 31), (14400, 61), (7200, 2), (7200, 31), (3600, 61), (1800, 61),
                                          (360, 61), (9000, 2), (16384, 2)])
def test_weight_gradient_from_stored_spectra(rosar, n_az, n_scans):
    import torch
    rng = np.random.default_rng(n_az + n_scans)
    n_rng, K = 5, 12
    o = (np.sort(rng.choice(600 if n_az > 600 else n_az, K, replace=False)) - 100).astype(np.int32)
    S, g, w = _c(rng, n_scans, n_rng, n_az), _c(rng, n_scans, n_rng, n_az), _c(rng, n_rng, K)
    tS, tg, tw, to = (torch.from_numpy(x).cuda() for x in (S, g, w, o))
    H = rosar.azimuth_plan(tw, to, n_az)
    X, G = torch.empty_like(tS), torch.empty_like(tS)
    rosar.sparse_azimuth_fft_scans_ex(tS, H, spectrum=X)
    rosar.sparse_azimuth_fft_scans_ex(tg, H, adjoint=True, spectrum=G)
    got = rosar.azimuth_weight_grad_spectra(G, X, to, K).cpu().numpy()
    ref = sum(O.sparse_azimuth_adjoint_w(g[s], S[s], o) for s in range(n_scans))
    assert np.linalg.norm(got - ref) < 1e-5 * np.linalg.norm(ref)      # the bar of the gradients' parity test
