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


# errors: the window of two rows holds the chunks of 200 pulses of 800, not those of 264 or 400; nominal: 32 rows of 36
# pulses are summed directly, 40 rows or 64 pulses go through transforms
@pytest.mark.parametrize("n_az,L,n_rng,M,errors", [(800, 512, 511, 200, True), (800, 512, 511, 264, True),
                                                   (800, 512, 512, 400, True), (1800, 64, 32, 36, False),
                                                   (1800, 64, 40, 36, False), (1800, 64, 36, 64, False)])
def test_back_projection(rosar, n_az, L, n_rng, M, errors):
    import oracle as O
    import torch
    rng = np.random.default_rng(n_az + M)
    S = _c(rng, L, n_az)
    r = synth.TINY.radar
    api = rosar.Radar(r.fc, r.slope, r.t_sample(L), r.t_start, r.r0, r.c)
    rad = O.Radar(fc=r.fc, slope=r.slope, t_s=r.t_sample(L), t_start=r.t_start, r0=r.r0, c=r.c)
    dphi = np.deg2rad(0.05 * rng.standard_normal(n_az)).astype(np.float32) if errors else None
    dr = (1e-3 * rng.standard_normal(n_az)).astype(np.float32) if errors else None
    dev = [None if x is None else torch.from_numpy(x).cuda() for x in (dphi, dr)]
    got = rosar.bpa(torch.from_numpy(S).cuda(), api, n_rng, M, dphi=dev[0], dr=dev[1]).cpu().numpy()
    rows = np.concatenate([rng.integers(0, n_rng, 60), [0, 0, 1, n_rng - 1, n_rng - 2]])
    th = np.concatenate([rng.integers(0, n_az, 60), [0, n_az - 1, 5, 7, n_az // 2]])
    kw = {} if not errors else {"dphi": dphi.astype(np.float64), "dr": dr.astype(np.float64)}
    ref = O.bpa_pixels(S, rad, n_az, M, rows, th, **kw)
    assert np.linalg.norm(got[rows, th] - ref) <= 1e-4 * np.linalg.norm(ref)       # the parity tests' bar


# launched over range compression's tail (one CTA an SM, short CTAs, many CTAs) or after it (2047 x 256, 128 taps)
@pytest.mark.parametrize("n_az,L,K", [(360, 64, 16), (2047, 256, 16), (2047, 256, 128), (3607, 256, 64), (541, 1024, 64)])
def test_gather_image_equals_its_two_steps(rosar, n_az, L, K):
    import torch
    rng = np.random.default_rng(n_az + K)
    raw, w = torch.from_numpy(_c(rng, n_az, L)).cuda(), torch.from_numpy(_c(rng, L, K)).cuda()
    o = torch.from_numpy(rng.integers(-n_az, n_az, K).astype(np.int32)).cuda()
    win = torch.from_numpy(synth.hann_window(L)).cuda()
    S = rosar.range_compress(raw, win)
    want = rosar.sparse_azimuth(S, w, o)
    for _ in range(3):
        assert torch.equal(rosar.image(raw, win, w, o), want)


# rows of the compile-time lengths: H staged up to 456 rows, read in the fused step from 457 on (7200 and 14400: 152, 153)
@pytest.mark.parametrize("n_az,rows", [(360, 456), (360, 457), (1800, 456), (1800, 457), (3600, 456), (3600, 457),
                                       (7200, 152), (7200, 153), (14400, 153), (800, 304), (800, 305)])
def test_row_filter(rosar, n_az, rows):
    import oracle as O
    import torch
    rng = np.random.default_rng(n_az + rows)
    w = _c(rng, rows, 6)
    o = rng.integers(-n_az, n_az, 6).astype(np.int32)
    S = _c(rng, rows, n_az)
    tS, tw, to = (torch.from_numpy(x).cuda() for x in (S, w, o))
    H = rosar.azimuth_plan(tw, to, n_az)
    got = rosar.sparse_azimuth_fft(tS, H)
    for a in (0, 100, rows - 50):                    # few rows of it alone
        assert torch.equal(rosar.sparse_azimuth_fft(tS[a:a + 50].contiguous(), H[a:a + 50].contiguous()), got[a:a + 50])
    ref = O.sparse_azimuth(S[-3:], w[-3:], o)
    assert np.linalg.norm(got[-3:].cpu().numpy() - ref) <= 5e-6 * np.linalg.norm(ref)      # the filter's bar
    X = torch.empty_like(tS)[None]
    G = torch.empty_like(X)
    rosar.sparse_azimuth_fft_scans_ex(tS[None], H, spectrum=X)
    rosar.sparse_azimuth_fft_scans_ex(got[None], H, adjoint=True, spectrum=G)
    grad = rosar.azimuth_weight_grad_spectra(G, X, to, 6).cpu().numpy()
    ref = O.sparse_azimuth_adjoint_w(got[-3:].cpu().numpy(), S[-3:], o)
    assert np.linalg.norm(grad[-3:] - ref) <= 1e-5 * np.linalg.norm(ref)                   # the gradients' bar
