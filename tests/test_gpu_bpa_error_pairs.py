"""Back-projection with supplied errors on grids large enough for the kernel of two rows a thread (608 CTAs): both
interpolations, odd row counts, chunks of offsets of every size, windows that cannot be bounded, errors that are NaN."""

import numpy as np
import pytest

import oracle as O
import synth

pytestmark = pytest.mark.gpu

TOL_IMAGE = 1e-4     # the relative-L2 bar of the parity tests


@pytest.fixture(scope="module")
def rosar():
    from paper_2309_08038_gb300 import build
    build.build()
    import paper_2309_08038_gb300 as r
    return r


def _errors(kind, rng, n_az, dR):
    dphi = np.deg2rad(0.05 * rng.standard_normal(n_az)).astype(np.float32)
    dr = (1e-3 * rng.standard_normal(n_az)).astype(np.float32)
    if kind == "far":            # pulses several bins out and some degrees off: their chunks' windows are not bounded
        dr[190:200] = np.float32(3.5 * dR)
        dphi[190:200] = np.float32(np.deg2rad(4.0))
        dr[700] = np.float32(-2.5 * dR)
        dr[n_az - 1] = np.float32(200 * dR)                     # bins past the last one read zero
    elif kind == "nan":
        dphi[7] = np.nan
        dr[1200] = np.nan
    return dphi, dr


# (n_az, L, n_rng, M): odd row counts (the last pair holds one), n_rng below and at L, a ragged azimuth tile, apertures of
# one pulse, one chunk of the largest size and one more, three chunks, and the whole ring
SIZES = [(2500, 128, 127, 60), (2500, 160, 129, 1), (2304, 256, 137, 256), (2500, 256, 135, 257), (3600, 128, 91, 600),
         (1300, 512, 203, 1300)]


@pytest.mark.parametrize("kind", ["small", "far", "nan"])
@pytest.mark.parametrize("interp", ["linear", "nearest"])
@pytest.mark.parametrize("n_az,L,n_rng,M", SIZES)
def test_pairs_of_rows_match_oracle(rosar, n_az, L, n_rng, M, interp, kind):
    import torch
    assert (n_az + 255) // 256 * ((n_rng + 1) // 2) >= 608
    rng = np.random.default_rng(n_az + M)
    S = (rng.standard_normal((L, n_az)) + 1j * rng.standard_normal((L, n_az))).astype(np.complex64)
    r = synth.TINY.radar
    api = rosar.Radar(r.fc, r.slope, r.t_sample(L), r.t_start, r.r0, r.c)
    rad = O.Radar(fc=r.fc, slope=r.slope, t_s=r.t_sample(L), t_start=r.t_start, r0=r.r0, c=r.c)
    dR = O.range_bin_spacing(rad, L)
    dphi, dr = _errors(kind, rng, n_az, dR)
    got = rosar.bpa(torch.from_numpy(S).cuda(), api, n_rng, M, interp=interp, dphi=torch.from_numpy(dphi).cuda(),
                    dr=torch.from_numpy(dr).cuda()).cpu().numpy()
    assert got.shape == (n_rng, n_az)
    d = np.arange(-(M // 2), M - M // 2)
    near = np.concatenate([np.arange(180, 210), np.arange(690, 710), np.arange(n_az - 5, n_az), np.arange(0, 10)])
    th = np.unique(np.concatenate([near, np.arange(0, n_az, 41)]))
    n = (th[:, None] + d[None, :]) % n_az
    read_nan = np.isnan(dphi[n] + dr[n]).any(1)
    e64, r64 = dphi.astype(np.float64), dr.astype(np.float64)
    checked = 0
    for row in (0, 1, 2, n_rng // 2, n_rng - 2, n_rng - 1):
        y = got[row, th]
        assert np.array_equal(np.isnan(y), read_nan), row
        keep = ~read_nan
        if interp == "nearest":      # a bin within 1e-3 of a tie may round either way
            x = O.slant_range(rad.r0 + row * dR, O.phase_centre_angle(th, n_az)[:, None], rad.r0 + r64[n],
                              O.phase_centre_angle(n, n_az) + e64[n]) / dR
            with np.errstate(invalid="ignore"):
                keep &= np.all(~(np.abs(x - np.floor(x) - 0.5) < 1e-3), axis=1)
        if not keep.any():
            continue
        t = th[keep]
        ref = O.bpa_pixels(S, rad, n_az, M, np.full(t.size, row), t, interp, dphi=e64, dr=r64)
        assert np.linalg.norm(y[keep] - ref) <= TOL_IMAGE * np.linalg.norm(ref), row
        checked += t.size
    # the whole ring reads every pulse: a NaN reaches every pixel, and a tie lies within reach of nearly all
    assert checked >= 20 or M == n_az
